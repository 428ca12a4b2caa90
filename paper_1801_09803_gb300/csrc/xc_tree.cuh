// xc_tree.cuh -- line index, ranges and the taking rule of the block-interpolated sweeps
// (FP32: xc_tree.cu, FP64: xc_tree64.cu).
#pragma once

#include "xc_batched.cuh"

namespace xc {

constexpr int TR_LEVELS = 3;
constexpr int TR_M = 16;                    // nodes per block
__device__ __host__ constexpr int tr_block(int lev) { return lev == 0 ? 64 : (lev == 1 ? 128 : 512); }
__device__ __host__ constexpr int tr_gap(int lev) { return lev == 0 ? 36 : (lev == 1 ? 72 : 284); }   // 0.55 B
constexpr int TR_T = 256;                   // threads per CTA
constexpr int TR_W = TR_T / 32;
constexpr int TR_CELL = 64;                 // grid steps per entry of the line index

struct TreeParams {
    LinesDev L;
    const int4 *geo;             // per line: integer grid position n, cut range ka..kb (inclusive), fraction f (bits)
    const float4 *recA, *recB;   // per (condition, line): profile constants (see line_consts); B: Voigt w4 only
    const CParam *cp;
    const GeomStats *gs;
    const unsigned *cell;        // cell[j]: first line with n >= cell0 + 64 j, j = 0..ncell
    int cell0, ncell;
    double *nodes;               // per condition: node sums of levels 0, 1, 2
    int nblk[TR_LEVELS], node_off[TR_LEVELS], nodes_per_cond;
    const double *mat;           // interpolation matrices (see TR_MAT_*)
    int c0, n_cond;              // conditions c0 .. c0 + n_cond - 1 of the call are in recA / recB
    size_t n;                    // lines
    int n_pts;
    int reach;                   // no line reaches a point farther than this many steps from its n
    int cover;                   // every line covers the points within this many steps (0: not known)
    int far;                     // 0: no blocks (profiles without far wings)
    int wpt;                     // warps per task (points)
    int wptl[TR_LEVELS], ncta[TR_LEVELS];   // nodes: warps per task and CTAs of each level
    double nu_A, step, cutoff;
    float inv_h, ext;            // ext: real distance of the outermost pole from the centre, per alpha (grid steps)
    int ext0;                    // ... plus this many steps
    float core;                  // radius of the points that need the full profile, per alpha
    const double *ghx, *ghw;
    int ngh;
    float gh_ext;                // bound of the Gauss-Hermite nodes
    double *sigma;               // [n_cond rows of the call][n_pts]
};

// interpolation matrices, destination index fastest: nodes of a 512-point block -> nodes of its
// eight 64-point blocks, of a 128-point block -> its two, of a 64-point block -> its points
constexpr int TR_MAT_512 = 0;                              // [8][16 source][16]
constexpr int TR_MAT_128 = 8 * TR_M * TR_M;                // [2][16 source][16]
constexpr int TR_MAT_PT = TR_MAT_128 + 2 * TR_M * TR_M;    // [16 source][64]
constexpr int TR_MAT = TR_MAT_PT + TR_M * 64;

// node m of a block of B points, in grid steps from its first point: Chebyshev nodes of
// [0, B - 1] rounded to 1/128, so that node - n is exact in FP32
__device__ __forceinline__ float tr_node(int B, int m) {
    return rintf(64.f * (float)(B - 1) * (1.f - cospif((float)(2 * m + 1) * (1.f / (2 * TR_M))))) * (1.f / 128.f);
}

// Gap (grid steps) beyond which a block ending at b1 takes a line: the same for all lines of
// a condition (alpha from an upper bound of the wavenumbers that reach the block), growing
// with the level and with the block's position, so a line taken by a block is taken by its
// children.  acoef: the condition's alpha / nu.
__device__ __forceinline__ int tr_radius(const TreeParams &p, float acoef, int gap, int b1) {
    const float nu = fmaxf(__double2float_ru(__dadd_rn(grid_x(p.nu_A, p.step, b1), p.cutoff)), 0.f);
    const float ah = __fmul_ru(__fmul_ru(__fmul_ru(acoef, 1.00001f), nu), p.inv_h);
    const int a = gap + p.ext0 + (int)ceilf(__fmul_ru(fminf(ah, 1e6f), p.ext));
    const int b = (int)ceilf(__fmul_ru(fminf(ah, 1e6f), p.core)) + 2;
    return max(a, b);
}

// a block [b0, b1] (b1c: clipped to the grid) with radius D takes a line
__device__ __forceinline__ bool tr_takes(const int4 &g, int b0, int b1, int b1c, int D) {
    return g.y <= b0 && g.z >= b1c && (g.x < b0 - D || g.x > b1 + D);
}

__device__ __forceinline__ unsigned tr_lower(const TreeParams &p, int v) {   // <= first line with n >= v
    return p.cell[min(max((v - p.cell0) >> 6, 0), p.ncell)];
}
__device__ __forceinline__ unsigned tr_upper(const TreeParams &p, int v) {   // >= first line with n >= v
    return p.cell[min(max((v - p.cell0 + (TR_CELL - 1)) >> 6, 0), p.ncell)];
}

// bits of the lanes k0..k1 (0 <= k0, k1 <= 31; none when k1 < k0)
__device__ __forceinline__ unsigned lanes_of(int k0, int k1) {
    return k1 < k0 ? 0u : (0xffffffffu >> (31 - (k1 - k0))) << k0;
}

struct Segs {
    unsigned s[4], e[4];
};

// Candidate lines of a block of a far level: positions that can cover it, outside its radius,
// without those its parent takes for certain.  Ranges are rounded outwards to index cells and
// kept disjoint; tr_takes decides per line.
__device__ __forceinline__ Segs tr_far_segs(const TreeParams &p, int b0, int b1, int D, bool has_parent, int p0,
                                            int p1, int Dp) {
    const int b1c = min(b1, p.n_pts - 1);
    const int a = b1c - p.reach, z = b0 - D;
    int e1 = z, s2 = z;
    if (has_parent) {
        e1 = min(z, max(a, p1 - p.cover));
        s2 = min(z, max(e1, p0 - Dp));
    }
    const int a2 = b1 + D + 1, z2 = b0 + p.reach + 1;
    int e3 = z2, s4 = z2;
    if (has_parent) {
        e3 = min(z2, p1 + Dp + 1);
        s4 = min(z2, max(e3, p0 + p.cover));
    }
    Segs g;
    g.s[0] = tr_lower(p, a);
    g.e[0] = max(g.s[0], a < e1 ? tr_upper(p, e1) : 0u);
    g.s[1] = max(g.e[0], tr_lower(p, s2));
    g.e[1] = max(g.s[1], s2 < z ? tr_upper(p, z) : 0u);
    g.s[2] = max(g.e[1], tr_lower(p, a2));
    g.e[2] = max(g.s[2], a2 < e3 ? tr_upper(p, e3) : 0u);
    g.s[3] = max(g.e[2], tr_lower(p, s4));
    g.e[3] = max(g.s[3], s4 < z2 ? tr_upper(p, z2) : 0u);
    return g;
}

// Candidate lines of the points s0..s1 inside the level-0 block [p0, p1] of radius Dp; far: lines that
// the block takes are left out
__device__ __forceinline__ Segs tr_point_segs(const TreeParams &p, bool far, int s0, int s1, int p0, int p1, int Dp) {
    const int a = s0 - p.reach, z = s1 + p.reach + 1;
    int e1 = a, s2 = a, e2 = z, s3 = z;
    if (far) {
        e1 = max(a, min(p0 - Dp, p1 - p.cover));
        s2 = max(e1, p0 - Dp);
        e2 = min(z, p1 + Dp + 1);
        s3 = min(z, max(e2, p0 + p.cover));
    }
    Segs g;
    g.s[0] = tr_lower(p, a);
    g.e[0] = max(g.s[0], a < e1 ? tr_upper(p, e1) : 0u);
    g.s[1] = max(g.e[0], tr_lower(p, s2));
    g.e[1] = max(g.s[1], s2 < e2 ? tr_upper(p, e2) : 0u);
    g.s[2] = max(g.e[1], tr_lower(p, s3));
    g.e[2] = max(g.s[2], s3 < z ? tr_upper(p, z) : 0u);
    g.s[3] = g.e[3] = g.e[2];
    return g;
}

// the FP32 sweep's interpolation matrices (TR_MAT doubles, see TR_MAT_*)
cudaError_t launch_tree_mat(double *mat, cudaStream_t s);
cudaError_t tree_mat(BatchedState *st, const double **mat, cudaStream_t s);   // the handle's copy

}  // namespace xc
