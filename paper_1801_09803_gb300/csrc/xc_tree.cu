// xc_tree.cu -- FP32 sweep with the far field of every line interpolated on blocks of the grid.
//
// Away from a line's centre its profile is a smooth function of the wavenumber, so on a
// block of B grid points that lies wholly inside the line's cut and far enough from the
// centre, its values at B points follow from its values at M = 16 Chebyshev nodes of the
// block.  Profiles of all lines are summed at the nodes, and the sums are interpolated to
// the points once.  Blocks of 512, 128 and 64 points are nested: a (line, point) pair
// belongs to the largest block that takes the line, and pairs that no block takes (near the
// centre, at the ends of the cut) are evaluated at the point itself.  A line with a cut of
// 2500 grid steps is evaluated at about 300 nodes and 220 points instead of 5000 points.
//
// Interpolation error.  The far profiles are analytic except at poles (branch points for
// the bin averages) near the line's centre, at real distance at most e (grid steps) from it:
// 0.85 alpha for w4's region I (poles at delta = +-0.849 alpha +- i gamma), the outermost
// shifted node for Gauss-Hermite sums, 0 for the Lorentzian.  With the pole at least
// 0.55 B from the block the degree-15 interpolant of 1/(x - s)^2 is within 1.6e-8 of every
// value (16 nodes; computed over all s: the worst is the nearest line, on the real axis),
// below the FP32 rounding of the profile itself.  A block takes a line when the gap between
// centre and block exceeds max(0.55 B + e, radius of w4's regions II to IV).
//
// Which block takes a pair is decided on integers (line position, cut range, block-wise
// radius), by the same expressions in every kernel, so each pair is counted exactly once.
// Gather form: one warp (or several, see warps_per_task) owns a block's nodes or 32 points
// and visits the lines of four ranges of the sorted list; no atomics, fixed order.
#include <math.h>
#include <stdio.h>

#include <algorithm>
#include <string>

#include "xc_batched.cuh"
#include "xc_f32.cuh"

namespace xc {

constexpr int TR_M = 16;                    // nodes per block
constexpr int TR_LEVELS = 3;
__device__ __host__ constexpr int tr_block(int lev) { return lev == 0 ? 64 : (lev == 1 ? 128 : 512); }
__device__ __host__ constexpr int tr_gap(int lev) { return lev == 0 ? 36 : (lev == 1 ? 72 : 284); }   // 0.55 B
constexpr int TR_T = 256;                   // threads per CTA
constexpr int TR_W = TR_T / 32;
constexpr int TR_FOLD = 4;                  // scanned chunks (32 lines) per FP32 partial sum at the nodes
                                            // (each chunk at the points, where one strong line can
                                            // dominate: 512 lines in one sum left 6e-7 of rounding)
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
    int wpt;                     // warps per task
    double nu_A, step, cutoff;
    float inv_h, ext;            // ext: real distance of the outermost pole from the centre, per alpha (grid steps)
    int ext0;                    // ... plus this many steps
    float core;                  // radius of the points that need the full profile, per alpha
    const double *ghx, *ghw;
    int ngh;
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

// Gap (grid steps) beyond which a block ending at b1 takes a line: the same for all lines
// (alpha from an upper bound of the wavenumbers that reach the block), growing with the
// level and with the block's position, so a line taken by a block is taken by its children
__device__ __forceinline__ int tr_radius(const TreeParams &p, int lev, int b1) {
    const float nu = fmaxf(__double2float_ru(__dadd_rn(grid_x(p.nu_A, p.step, b1), p.cutoff)), 0.f);
    const float ah = __fmul_ru(__fmul_ru(__uint_as_float(p.gs->acoef_bits), nu), p.inv_h);
    const int a = tr_gap(lev) + p.ext0 + (int)ceilf(__fmul_ru(fminf(ah, 1e6f), p.ext));
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

// Candidate lines of the points s0..s1 inside the level-0 block [p0, p1] of radius Dp
__device__ __forceinline__ Segs tr_point_segs(const TreeParams &p, int s0, int s1, int p0, int p1, int Dp) {
    const int a = s0 - p.reach, z = s1 + p.reach + 1;
    int e1 = a, s2 = a, e2 = z, s3 = z;
    if (p.far) {
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

template <int PROF>
__device__ __forceinline__ float tr_amplitude(const float4 &A) {
    return (PROF == XC_VOIGT_W4 || PROF == XC_VOIGT_GH_SAMPLED || PROF == XC_LORENTZ_BINNED) ? A.z
           : PROF == XC_VOIGT_GH_BINNED                                                     ? A.w
                                                                                            : A.y;
}
template <int PROF>
constexpr bool tr_pairs() { return PROF == XC_VOIGT_W4 || PROF == XC_LORENTZ; }

// two lines at one position per packed operation: region I of w4, or the Lorentzian
template <int PROF>
__device__ __forceinline__ f32x2 tr_pair_value(f32x2 u, const ulonglong2 &c0, const ulonglong2 &c1) {
    if (PROF == XC_VOIGT_W4) return mul2(fma2(c1.x, u, c1.y), rcp2(fma2(u, add2(u, c0.x), c0.y)));
    return mul2(c0.y, rcp2(add2(u, c0.x)));
}

// sum += acc, compensated
__device__ __forceinline__ void tr_fold(float &hi, float &lo, float &acc) {
    const float t = __fadd_rn(hi, acc), z = __fsub_rn(t, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, z)), __fsub_rn(acc, z)));
    hi = t;
    acc = 0.f;
}

// ---------------------------------------------------------------------------
// setup
// ---------------------------------------------------------------------------
__global__ void k_tree_prep(const CondDev *conds, int n_cond, GeomStats *gs) {
    __shared__ float s[32];
    float a = 0.f;
    for (int c = threadIdx.x; c < n_cond; c += 32)
        a = fmaxf(a, __double2float_ru(alpha_coef(conds[c].T, conds[c].mass_da) * (1.0 + 1e-6)));
    s[threadIdx.x] = a;
    __syncwarp();
    if (threadIdx.x == 0) {
        for (int i = 1; i < 32; ++i) a = fmaxf(a, s[i]);
        *gs = GeomStats{};
        gs->acoef_bits = __float_as_uint(a);
    }
}

// Line geometry in grid steps and the intensity statistics.  width_mult > 0: the cut of
// condition *cond; zero_k > 0: profiles that are exactly 0 in FP32 beyond
// zero_k alpha + zero_0 (grid steps) of the centre, alpha the largest of the conditions.
__global__ void __launch_bounds__(256) k_tree_geom(LinesDev L, size_t n, double nu_A, double step, int64_t n_pts,
                                                   double cutoff, double width_mult, const CondDev *cond,
                                                   float zero_k, double zero_0, int4 *geo, GeomStats *gs) {
    const double inv_h = 1.0 / step;
    float m1 = 0.f, m2 = 0.f, m3 = 0.f, m4 = 0.f, m5 = 0.f;
    double ac = 0.0, lnTr = 0.0, gsc = 0.0;
    CondDev c{};
    if (width_mult > 0.0) {
        c = *cond;
        ac = alpha_coef(c.T, c.mass_da);
        lnTr = log(c.T_ref / c.T);
        gsc = c.P / c.P_ref;
    }
    const double zk = (double)zero_k * (double)__uint_as_float(gs->acoef_bits);
    for (size_t l = (size_t)blockIdx.x * blockDim.x + threadIdx.x; l < n; l += (size_t)gridDim.x * blockDim.x) {
        const double nu = L.nu[l];
        const float gr = L.gamma_ref[l], nT = L.n_T[l];
        m3 = fmaxf(m3, __double2float_ru(fabs(nu)));
        m4 = fmaxf(m4, fabsf(gr));
        m5 = fmaxf(m5, fabsf(nT));
        double cut = cutoff;
        if (width_mult > 0.0) {
            const double ga = L.n_broad > 0 ? mixture_gamma64(L, l, c)
                                            : c.gamma_scale * (double)gr * exp(((double)nT + c.n_shift) * lnTr) * gsc;
            cut = fmin(width_mult * fmax(ac * nu, ga), cutoff);
        }
        if (zero_k > 0.f) cut = fmin(cut, zk * nu + zero_0 * step);
        const double d = (nu - nu_A) * inv_h;
        const double fl = floor(d);
        const double flc = fmin(fmax(fl, -1073741824.0), 1073741824.0);
        int64_t ka, kb;
        line_k_range(nu, cut, nu_A, step, inv_h, n_pts, &ka, &kb);
        if (kb < ka) { ka = 1; kb = 0; }
        geo[l] = make_int4((int)flc, (int)i64min(i64max(ka, -1), (int64_t)0x7fffffff),
                           (int)i64min(i64max(kb, -1), (int64_t)0x7fffffff), __float_as_int((float)(d - fl)));
        const float gA = (float)L.g_up[l] * L.A[l];
        const float nuf = (float)nu;
        m1 = fmaxf(m1, gA / (nuf * nuf));
        m2 = fmaxf(m2, gA / nuf);
    }
    for (int o = 16; o > 0; o >>= 1) {
        m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, o));
        m2 = fmaxf(m2, __shfl_xor_sync(0xffffffffu, m2, o));
        m3 = fmaxf(m3, __shfl_xor_sync(0xffffffffu, m3, o));
        m4 = fmaxf(m4, __shfl_xor_sync(0xffffffffu, m4, o));
        m5 = fmaxf(m5, __shfl_xor_sync(0xffffffffu, m5, o));
    }
    if ((threadIdx.x & 31) == 0) {
        if (isfinite(m1)) atomicMax(&gs->gA_nu2_bits, __float_as_uint(m1));
        if (isfinite(m2)) atomicMax(&gs->gA_nu_bits, __float_as_uint(m2));
        atomicMax(&gs->nu_bits, __float_as_uint(m3));   // non-negative floats: integer order
        atomicMax(&gs->gref_bits, __float_as_uint(m4));
        atomicMax(&gs->nT_bits, __float_as_uint(m5));
    }
}

// Lagrange basis polynomial of node m (of a block of B points) at x, from the nodes as rounded
__device__ double tr_basis(int B, int m, double x) {
    const double xm = (double)tr_node(B, m);
    double num = 1.0, den = 1.0;
    for (int j = 0; j < TR_M; ++j) {
        if (j == m) continue;
        const double xj = (double)tr_node(B, j);
        // scaled by the half-length so that the products stay near 1
        const double s = 4.0 / (double)B;
        num *= (x - xj) * s;
        den *= (xm - xj) * s;
    }
    return num / den;
}

// block 0: per-condition constants; block 1..: line index, then the interpolation matrices
__global__ void __launch_bounds__(256) k_tree_setup(TreeParams p, const CondDev *conds, int n_cond, CParam *cp,
                                                    int quantity, const unsigned *gmax, unsigned *cell, double *mat) {
    if (blockIdx.x == 0) {
        for (int c = threadIdx.x; c < n_cond; c += 256)
            cp[c] = make_cparam(c, conds, p.gs, p.step, quantity, gmax, 4.f, 0);
        return;
    }
    const int i = (blockIdx.x - 1) * 256 + threadIdx.x;
    if (i <= p.ncell) {
        const int v = p.cell0 + TR_CELL * i;
        size_t a = 0, b = p.n;
        while (a < b) {
            const size_t m = a + ((b - a) >> 1);
            if (p.geo[m].x < v) a = m + 1; else b = m;
        }
        cell[i] = (unsigned)a;
    }
    const int k = i - (p.ncell + 1);
    if (!p.far || k < 0 || k >= TR_MAT) return;
    if (k < TR_MAT_128) {
        const int j = k / (TR_M * TR_M), s = (k / TR_M) % TR_M, d = k % TR_M;
        mat[k] = tr_basis(512, s, (double)(64 * j) + (double)tr_node(64, d));
    } else if (k < TR_MAT_PT) {
        const int q = k - TR_MAT_128, j = q / (TR_M * TR_M), s = (q / TR_M) % TR_M, d = q % TR_M;
        mat[k] = tr_basis(128, s, (double)(64 * j) + (double)tr_node(64, d));
    } else {
        const int q = k - TR_MAT_PT;
        mat[k] = tr_basis(64, q / 64, (double)(q % 64));
    }
}

// profile constants of every (condition, line) of the group
template <int PROF, bool EXT>
__global__ void __launch_bounds__(256) k_tree_recs(TreeParams p, float4 *recA, float4 *recB) {
    const int c = blockIdx.y;
    const CParam cp = p.cp[p.c0 + c];
    const float h = (float)p.step;
    for (size_t l = (size_t)blockIdx.x * 256 + threadIdx.x; l < p.n; l += (size_t)gridDim.x * 256) {
        float4 A, B = make_float4(0.f, 0.f, 0.f, -1.f), S;
        float t2;
        line_consts<PROF, EXT>(p.L, l, cp, h, p.inv_h, &A, &B, &t2, &S);
        recA[(size_t)c * p.n + l] = A;
        if (PROF == XC_VOIGT_W4) recB[(size_t)c * p.n + l] = B;
    }
}

// ---------------------------------------------------------------------------
// far levels: sums at the nodes.  A warp holds 16 nodes twice: its half-warps take different
// lines.  Per 32 scanned lines the accepted ones are compacted into shared memory, pairs of
// lines interleaved for the packed arithmetic; one iteration of the loop takes 4 lines.
// ---------------------------------------------------------------------------
template <int PROF>
__global__ void __launch_bounds__(TR_T) k_tree_nodes(TreeParams p) {
    constexpr int PAIR = tr_pairs<PROF>() ? (PROF == XC_VOIGT_W4 ? 3 : 2) : 2;   // 16-byte words per pair
    __shared__ float4 sL[TR_W][tr_pairs<PROF>() ? 16 * PAIR : 48];   // non-pairs: 24 bytes a line
    __shared__ float sX[64], sW[64];
    __shared__ float2 sRed[TR_W][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, half = lane >> 4;
    if (p.ngh > 0) {
        if (threadIdx.x < p.ngh) {
            sX[threadIdx.x] = (float)p.ghx[threadIdx.x];
            sW[threadIdx.x] = (float)p.ghw[threadIdx.x];
        }
        __syncthreads();
    }
    const int wpt = p.wpt, part = warp % wpt;
    int task = blockIdx.x * (TR_W / wpt) + warp / wpt;
    const int c = blockIdx.y;
    int lev = 2;   // the largest blocks have the most lines: first
    if (task >= p.nblk[2]) {
        task -= p.nblk[2];
        lev = 1;
        if (task >= p.nblk[1]) {
            task -= p.nblk[1];
            lev = 0;
        }
    }
    const bool live = task < p.nblk[lev];
    float hi = 0.f, lo = 0.f;
    if (live) {
        const int B = tr_block(lev), b0 = task * B, b1 = b0 + B - 1, b1c = min(b1, p.n_pts - 1);
        const int D = tr_radius(p, lev, b1);
        const bool up = lev < 2;
        const int PB = up ? tr_block(lev + 1) : 1;
        const int p0 = up ? b0 / PB * PB : 0, p1 = p0 + PB - 1, p1c = min(p1, p.n_pts - 1);
        const int Dp = up ? tr_radius(p, lev + 1, p1) : 0;
        const Segs sg = tr_far_segs(p, b0, b1, D, up, p0, p1, Dp);
        const float x = tr_node(B, lane & 15);
        const f32x2 x2 = pk2(x, x);
        const float4 *recA = p.recA + (size_t)c * p.n;
        float4 *buf = sL[warp];
        f32x2 acc2 = 0ull;
        float acc = 0.f;
        int in_fold = 0;
#pragma unroll 1
        for (int k = 0; k < 4; ++k) {
            const unsigned e = sg.e[k];
            unsigned i = sg.s[k] + 32u * part;
            int4 g = make_int4(0, 1, 0, 0);
            if (i + lane < e) g = p.geo[i + lane];
#pragma unroll 1
            for (; i < e; i += 32u * wpt) {
                const unsigned l = i + lane;
                int4 gn = make_int4(0, 1, 0, 0);
                if (l + 32u * wpt < e) gn = p.geo[l + 32u * wpt];
                bool ok = l < e && tr_takes(g, b0, b1, b1c, D) && !(up && tr_takes(g, p0, p1, p1c, Dp));
                float4 A = make_float4(0.f, 0.f, 0.f, 0.f);
                if (ok) {
                    A = recA[l];
                    ok = tr_amplitude<PROF>(A) != 0.f;
                }
                const unsigned m = __ballot_sync(0xffffffffu, ok);
                const int cnt = __popc(m);
                if (cnt) {
                    const int pad = tr_pairs<PROF>() ? 4 : 2;
                    int slot = __popc(m & ((1u << lane) - 1u));
                    float n = (float)(g.x - b0), f = __int_as_float(g.w);
                    bool put = ok;
                    if (!ok) {   // lanes that fill the last iteration with lines of amplitude 0
                        const int z = __popc(~m & ((1u << lane) - 1u));
                        put = z < ((cnt + pad - 1) / pad * pad - cnt);
                        slot = cnt + z;
                        n = -1e4f;
                        f = 0.f;
                        A = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (PROF == XC_VOIGT_GH_BINNED) A.y = A.z = 1.f;
                        if (PROF == XC_LORENTZ_BINNED) A.x = A.y = 1.f;
                        if (PROF == XC_VOIGT_GH_SAMPLED) A.y = 1.f;
                    }
                    if (put) {
                        float *q = reinterpret_cast<float *>(buf);
                        if (tr_pairs<PROF>()) {
                            q += (slot >> 1) * (4 * PAIR) + (slot & 1);
                            q[0] = n;
                            q[2] = f;
                            q[4] = A.x;
                            q[6] = A.y;
                            if (PROF == XC_VOIGT_W4) {
                                q[8] = A.z;
                                q[10] = A.w;
                            }
                        } else {
                            // one line per 24 bytes: n, f, constants
                            reinterpret_cast<float2 *>(q)[slot * 3] = make_float2(n, f);
                            reinterpret_cast<float2 *>(q)[slot * 3 + 1] = make_float2(A.x, A.y);
                            reinterpret_cast<float2 *>(q)[slot * 3 + 2] = make_float2(A.z, A.w);
                        }
                    }
                    __syncwarp();
                    if (tr_pairs<PROF>()) {
#pragma unroll 2
                        for (int j = half; 2 * j < cnt; j += 2) {
                            const ulonglong2 *q = reinterpret_cast<const ulonglong2 *>(buf + j * PAIR);
                            const ulonglong2 nf = q[0], c0 = q[1];
                            ulonglong2 c1 = c0;
                            if (PROF == XC_VOIGT_W4) c1 = q[2];
                            const f32x2 d = sub2(sub2(x2, nf.x), nf.y);
                            const f32x2 u = mul2(d, d);
                            if (PROF == XC_VOIGT_W4)
                                acc2 = fma2(fma2(c1.x, u, c1.y), rcp2(fma2(u, add2(u, c0.x), c0.y)), acc2);
                            else
                                acc2 = fma2(c0.y, rcp2(add2(u, c0.x)), acc2);
                        }
                    } else {
                        for (int j = half; j < cnt; j += 2) {
                            const float2 *q = reinterpret_cast<const float2 *>(buf) + j * 3;
                            const float2 nf = q[0], a01 = q[1], a23 = q[2];
                            const float d = (x - nf.x) - nf.y;
                            acc += contrib_single<PROF>(d * d, d, make_float4(a01.x, a01.y, a23.x, a23.y),
                                                        make_float4(0.f, 0.f, 0.f, -1.f), sX, sW, p.ngh);
                        }
                    }
                    __syncwarp();
                    if (++in_fold == TR_FOLD) {
                        if (tr_pairs<PROF>()) {
                            acc = lo2(acc2) + lo2((acc2 >> 32) | (acc2 << 32));
                            acc2 = 0ull;
                        }
                        tr_fold(hi, lo, acc);
                        in_fold = 0;
                    }
                }
                g = gn;
            }
        }
        if (tr_pairs<PROF>()) acc = lo2(acc2) + lo2((acc2 >> 32) | (acc2 << 32));
        tr_fold(hi, lo, acc);
    }
    // the half-warps' (and the task's warps') sums, in a fixed order
    double v = (double)hi + (double)lo;
    v += __shfl_xor_sync(0xffffffffu, v, 16);
    if (wpt > 1) {
        double *red = reinterpret_cast<double *>(sRed);
        __syncthreads();
        red[warp * 32 + lane] = v;
        __syncthreads();
        if (part == 0)
            for (int w = 1; w < wpt; ++w) v += red[(warp + w) * 32 + lane];
    }
    if (live && part == 0 && half == 0)
        p.nodes[(size_t)c * p.nodes_per_cond + p.node_off[lev] + task * TR_M + lane] = v;
}

// ---------------------------------------------------------------------------
// points: the pairs no block takes, plus the interpolated sums.  A warp owns 32 points.  Lines
// whose full-profile zone cannot reach the points go in packed pairs (region I, masked by the
// cut), the others one by one with w4's regions per point.
// ---------------------------------------------------------------------------
template <int PROF>
__global__ void __launch_bounds__(TR_T) k_tree_points(TreeParams p) {
    constexpr bool W4 = PROF == XC_VOIGT_W4;
    __shared__ float4 sF[TR_W][tr_pairs<PROF>() ? 16 * 4 : 1];   // pairs: n, f | cut ranges | constants
    __shared__ float4 sC[TR_W][32 * (W4 ? 3 : 2)];               // singles: n, f, ka, kb | A | B
    __shared__ float sX[64], sW[64];
    __shared__ double sRed[TR_W][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (p.ngh > 0) {
        if (threadIdx.x < p.ngh) {
            sX[threadIdx.x] = (float)p.ghx[threadIdx.x];
            sW[threadIdx.x] = (float)p.ghw[threadIdx.x];
        }
        __syncthreads();
    }
    const int wpt = p.wpt, part = warp % wpt;
    const int task = blockIdx.x * (TR_W / wpt) + warp / wpt;
    const int c = blockIdx.y;
    const int s0 = task * 32, s1 = s0 + 31;
    const bool live = s0 < p.n_pts;
    float hi = 0.f, lo = 0.f;
    if (live) {
        const int p0 = s0 & ~63, p1 = p0 + 63, p1c = min(p1, p.n_pts - 1);
        const int Dp = p.far ? tr_radius(p, 0, p1) : 0;
        // points within this of a line may need its full profile (w4's regions II to IV)
        int core = 0;
        if (W4) {
            const float nu = fmaxf(__double2float_ru(__dadd_rn(grid_x(p.nu_A, p.step, p1), p.cutoff)), 0.f);
            core = (int)ceilf(__fmul_ru(fminf(__fmul_ru(__fmul_ru(__uint_as_float(p.gs->acoef_bits), nu), p.inv_h), 1e6f),
                                        p.core)) + 2;
        }
        const Segs sg = tr_point_segs(p, s0, s1, p0, p1, Dp);
        const float x = (float)lane;
        const f32x2 x2 = pk2(x, x);
        const float4 *recA = p.recA + (size_t)c * p.n;
        const float4 *recB = p.recB + (size_t)c * p.n;
        float4 *bufF = sF[warp], *bufC = sC[warp];
        f32x2 acc2 = 0ull;
        float acc = 0.f;
#pragma unroll 1
        for (int k = 0; k < 3; ++k) {
            const unsigned e = sg.e[k];
            unsigned i = sg.s[k] + 32u * part;
            int4 g = make_int4(0, 1, 0, 0);
            if (i + lane < e) g = p.geo[i + lane];
#pragma unroll 1
            for (; i < e; i += 32u * wpt) {
                const unsigned l = i + lane;
                int4 gn = make_int4(0, 1, 0, 0);
                if (l + 32u * wpt < e) gn = p.geo[l + 32u * wpt];
                bool ok = l < e && g.y <= s1 && g.z >= s0 && g.y <= g.z &&
                          !(p.far && tr_takes(g, p0, p1, p1c, Dp));
                const bool cen = !tr_pairs<PROF>() || (W4 && g.x >= s0 - core && g.x <= s1 + core);
                float4 A = make_float4(0.f, 0.f, 0.f, 0.f), Bv = make_float4(0.f, 0.f, 0.f, -1.f);
                if (ok) {
                    A = recA[l];
                    if (W4 && cen) Bv = recB[l];
                    ok = W4 && cen ? Bv.z != 0.f : tr_amplitude<PROF>(A) != 0.f;
                }
                const unsigned mc = __ballot_sync(0xffffffffu, ok && cen);
                const unsigned mf = tr_pairs<PROF>() ? __ballot_sync(0xffffffffu, ok && !cen) : 0u;
                if (mc | mf) {
                    const unsigned below = (1u << lane) - 1u;
                    const float n = (float)(g.x - s0), f = __int_as_float(g.w);
                    const int ka = max(g.y - s0, 0), kb = min(g.z - s0, 31);
                    if (ok && cen) {
                        float4 *q = bufC + __popc(mc & below) * (W4 ? 3 : 2);
                        q[0] = make_float4(n, f, __int_as_float(ka), __int_as_float(kb));
                        q[1] = A;
                        if (W4) q[2] = Bv;
                    }
                    if (tr_pairs<PROF>()) {
                        const int cnt = __popc(mf);
                        const bool fill = !(ok && !cen) && (cnt & 1) && __popc(~mf & below) == 0;
                        if ((ok && !cen) || fill) {
                            const int slot = fill ? cnt : __popc(mf & below);
                            float *q = reinterpret_cast<float *>(bufF) + (slot >> 1) * 16 + (slot & 1);
                            q[0] = fill ? -1e4f : n;
                            q[2] = fill ? 0.f : f;
                            q[4] = __int_as_float(fill ? 0 : ka);
                            q[6] = __int_as_float(fill ? -1 : kb - ka);
                            q[8] = fill ? 0.f : A.x;
                            q[10] = fill ? 0.f : A.y;
                            if (W4) {
                                q[12] = fill ? 0.f : A.z;
                                q[14] = fill ? 0.f : A.w;
                            }
                        }
                    }
                    __syncwarp();
                    if (tr_pairs<PROF>()) {
                        const int cnt = __popc(mf);
#pragma unroll 2
                        for (int j = 0; 2 * j < cnt; ++j) {
                            const ulonglong2 *q = reinterpret_cast<const ulonglong2 *>(bufF + j * 4);
                            const ulonglong2 nf = q[0], c0 = q[2];
                            ulonglong2 c1 = c0;
                            if (W4) c1 = q[3];
                            const int4 kk = reinterpret_cast<const int4 *>(bufF + j * 4)[1];   // ka1 ka2 w1 w2
                            const f32x2 d = sub2(sub2(x2, nf.x), nf.y);
                            const f32x2 v = tr_pair_value<PROF>(mul2(d, d), c0, c1);
                            float v1, v2;
                            upk2(v, v1, v2);
                            v1 = lane - kk.x >= 0 && lane - kk.x <= kk.z ? v1 : 0.f;
                            v2 = lane - kk.y >= 0 && lane - kk.y <= kk.w ? v2 : 0.f;
                            acc2 = add2(acc2, pk2(v1, v2));
                        }
                    }
                    const int cnt = __popc(mc);
                    for (int j = 0; j < cnt; ++j) {
                        // a strong line's value in the sum makes the next ones' rounding: 16 a sum
                        if ((j & 15) == 15) tr_fold(hi, lo, acc);
                        const float4 *q = bufC + j * (W4 ? 3 : 2);
                        const float4 t = q[0], a = q[1];
                        const float d = (x - t.x) - t.y, u = d * d;
                        if (lane < __float_as_int(t.z) || lane > __float_as_int(t.w)) continue;
                        if (W4) {
                            const float4 b = q[2];
                            const float xx = b.x * fabsf(d), s = xx + b.y;
                            if (u >= b.w)
                                acc = fmaf(fmaf(a.z, u, a.w), rcp_approx(fmaf(u, u + a.x, a.y)), acc);
                            else
                                acc = fmaf(b.z, s >= 15.f ? w4_region1_re(xx, b.y)
                                                          : (s >= 5.5f ? w4_region2_re(xx, b.y) : w4_region34_re(xx, b.y)),
                                           acc);
                        } else {
                            acc += contrib_single<PROF>(u, d, a, make_float4(0.f, 0.f, 0.f, -1.f), sX, sW, p.ngh);
                        }
                    }
                    __syncwarp();
                    if (tr_pairs<PROF>()) {
                        acc += lo2(acc2) + lo2((acc2 >> 32) | (acc2 << 32));
                        acc2 = 0ull;
                    }
                    tr_fold(hi, lo, acc);
                }
                g = gn;
            }
        }
    }
    double v = (double)hi + (double)lo;
    if (wpt > 1) {
        __syncthreads();
        sRed[warp][lane] = v;
        __syncthreads();
        if (part == 0)
            for (int w = 1; w < wpt; ++w) v += sRed[warp + w][lane];
    }
    if (!live || part != 0) return;
    if (p.far) {
        // node sums of the enclosing blocks, brought down to the level-0 block and to the points
        const double *nd = p.nodes + (size_t)c * p.nodes_per_cond;
        const int j = s0 >> 6, m = lane & 15;
        double t = 0.0;
        if (lane < 16) {
            const double *src = nd + p.node_off[2] + (j >> 3) * TR_M, *w = p.mat + TR_MAT_512 + (j & 7) * (TR_M * TR_M) + m;
#pragma unroll
            for (int s = 0; s < TR_M; ++s) t = fma(w[s * TR_M], src[s], t);
            t += nd[p.node_off[0] + j * TR_M + m];
        } else {
            const double *src = nd + p.node_off[1] + (j >> 1) * TR_M, *w = p.mat + TR_MAT_128 + (j & 1) * (TR_M * TR_M) + m;
#pragma unroll
            for (int s = 0; s < TR_M; ++s) t = fma(w[s * TR_M], src[s], t);
        }
        t += __shfl_xor_sync(0xffffffffu, t, 16);
        const double *w = p.mat + TR_MAT_PT + (s0 & 63) + lane;
#pragma unroll
        for (int s = 0; s < TR_M; ++s) v = fma(w[s * 64], __shfl_sync(0xffffffffu, t, s), v);
    }
    const int k = s0 + lane;
    if (k < p.n_pts) {
        const CParam &cp = p.cp[p.c0 + c];
        p.sigma[(size_t)cp.row * (size_t)p.n_pts + k] = v * cp.inv_scale;
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
namespace {

#define TR_TRY(call)                                                                            \
    do {                                                                                        \
        cudaError_t _e = (call);                                                                \
        if (_e == cudaErrorMemoryAllocation) {                                                  \
            cudaGetLastError();                                                                 \
            set_error("device allocation failed: %s", #call);                                   \
            return XC_ENOMEM;                                                                   \
        }                                                                                       \
        if (_e != cudaSuccess) {                                                                \
            set_error("%s failed: %s (%s:%d)", #call, cudaGetErrorString(_e), __FILE__, __LINE__); \
            return XC_ECUDA;                                                                    \
        }                                                                                       \
    } while (0)

typedef void (*RecFn)(TreeParams, float4 *, float4 *);
typedef void (*TaskFn)(TreeParams);
struct ProfFns {
    RecFn rec, rec_ext;
    TaskFn nodes, points;
};

#define TR_FNS(P) {k_tree_recs<P, false>, k_tree_recs<P, true>, k_tree_nodes<P>, k_tree_points<P>}
bool fns_of(int profile, ProfFns *f) {
    switch (profile) {
    case XC_DOPPLER: *f = ProfFns TR_FNS(XC_DOPPLER); return true;
    case XC_LORENTZ: *f = ProfFns TR_FNS(XC_LORENTZ); return true;
    case XC_VOIGT_W4: *f = ProfFns TR_FNS(XC_VOIGT_W4); return true;
    case XC_VOIGT_GH_BINNED: *f = ProfFns TR_FNS(XC_VOIGT_GH_BINNED); return true;
    case XC_VOIGT_GH_SAMPLED: *f = ProfFns TR_FNS(XC_VOIGT_GH_SAMPLED); return true;
    case XC_DOPPLER_BINNED: *f = ProfFns TR_FNS(XC_DOPPLER_BINNED); return true;
    case XC_LORENTZ_BINNED: *f = ProfFns TR_FNS(XC_LORENTZ_BINNED); return true;
    default: return false;
    }
}

bool is_doppler(int profile) { return profile == XC_DOPPLER || profile == XC_DOPPLER_BINNED; }

// warps per task: several where the tasks alone would leave the SMs with few warps
int warps_per_task(int64_t tasks) {
    int w = 1;
    while (w < TR_W && tasks * w < 152 * 32) w *= 2;
    return w;
}

constexpr size_t kMaxRecBytes = (size_t)24 << 30;   // profile constants held at a time

}  // namespace

bool tree_takes(const BatchedArgs &a) {
    ProfFns f;
    return fns_of(a.opts.profile, &f) && a.opts.cutoff / a.grid.step < (double)(1 << 20) && a.grid.n < ((int64_t)1 << 30) &&
           a.n_lines < ((size_t)15 << 28);
}

xc_status tree_run(BatchedState *st, const BatchedArgs &a, int64_t *launches) {
    cudaStream_t s = a.stream;
    const size_t n = a.n_lines;
    const bool per_cond = a.opts.width_mult > 0.0;
    ProfFns fn;
    fns_of(a.opts.profile, &fn);
    const bool ext = a.opts.quantity != XC_ABSORPTION || a.opts.threshold != XC_THRESHOLD_NONE || a.L.n_broad > 0;
    const bool w4 = a.opts.profile == XC_VOIGT_W4;
    const int nc_all = a.n_cond;
    const int nc_pass = per_cond ? 1 : nc_all;             // conditions that share a line geometry
    int cg = (int)std::min<size_t>((size_t)nc_pass, std::max<size_t>(1, kMaxRecBytes / (n * (w4 ? 32 : 16))));

    TreeParams p;
    p.L = a.L;
    p.n = n;
    p.n_pts = (int)a.grid.n;
    p.nu_A = a.grid.nu_A;
    p.step = a.grid.step;
    p.cutoff = a.opts.cutoff;
    p.inv_h = (float)(1.0 / a.grid.step);
    const bool dop = is_doppler(a.opts.profile);
    p.far = dop ? 0 : 1;
    p.reach = (int)ceil(a.opts.cutoff / a.grid.step) + 2;
    p.cover = per_cond || dop ? 0 : std::max(0, (int)floor(a.opts.cutoff / a.grid.step) - 2);
    p.core = w4 ? 18.05f : 0.f;
    p.ext = 0.f;
    p.ext0 = 1;
    p.ngh = 0;
    p.ghx = a.ghx;
    p.ghw = a.ghw;
    if (w4) {
        p.ext = 0.86f;
        p.ext0 = 2;
    } else if (a.opts.profile == XC_LORENTZ_BINNED) {
        p.ext0 = 2;
    } else if (a.opts.profile == XC_VOIGT_GH_BINNED || a.opts.profile == XC_VOIGT_GH_SAMPLED) {
        p.ngh = a.opts.n_gh;
        p.ext = (float)(sqrt(2.0 * a.opts.n_gh + 2.0) / 0.83255) * 1.001f;   // nodes lie within sqrt(2 n + 2)
        p.ext0 = 3;
    }
    // Doppler profiles are exactly 0 in FP32 beyond these radii: 2^-x and erfc(x) underflow
    const float zero_k = a.opts.profile == XC_DOPPLER ? 12.3f : (dop ? 12.4f : 0.f);
    if (dop) {
        double am = 0.0;
        for (int c = 0; c < nc_all; ++c) am = std::max(am, alpha_coef(a.conds_host[c].T, a.conds_host[c].mass_da));
        const double top = a.grid.nu_A + a.grid.step * (double)a.grid.n + a.opts.cutoff;
        const double r = ceil((double)zero_k * am * 1.001 * std::max(top, 0.0) / a.grid.step) + 4.0;
        if (r < (double)p.reach) p.reach = (int)r;
    }
    p.cell0 = -TR_CELL * ((p.reach + 2 * TR_CELL) / TR_CELL);
    p.ncell = (int)(((int64_t)p.n_pts - p.cell0 + p.reach + 2 * TR_CELL) / TR_CELL);
    int off = 0;
    for (int lev = TR_LEVELS - 1; lev >= 0; --lev) {
        p.nblk[lev] = p.far ? (p.n_pts + tr_block(lev) - 1) / tr_block(lev) : 0;
        p.node_off[lev] = off;
        off += p.nblk[lev] * TR_M;
    }
    p.nodes_per_cond = off;

    size_t o = 0;
    auto carve = [&](size_t bytes) { size_t r = o; o += (bytes + 255) & ~size_t(255); return r; };
    // (the caller falls back to the tiled kernels when this does not fit in device memory)
    const size_t o_gs = carve(sizeof(GeomStats)), o_cp = carve((size_t)nc_pass * sizeof(CParam));
    const size_t o_cell = carve((size_t)(p.ncell + 1) * 4), o_mat = carve(TR_MAT * 8);
    const size_t o_nodes = carve((size_t)cg * p.nodes_per_cond * 8);
    const size_t o_geo = carve(n * sizeof(int4));
    const size_t o_A = carve((size_t)cg * n * 16), o_B = carve(w4 ? (size_t)cg * n * 16 : 16);
    size_t o_keep = 0, o_glc = 0, o_gmax = 0;
    if (a.opts.threshold != XC_THRESHOLD_NONE) o_keep = carve(n * (size_t)((nc_pass + 31) / 32) * 4);
    if (a.L.n_broad > 0) {
        o_glc = carve(n * (size_t)nc_pass * 4);
        o_gmax = carve((size_t)nc_pass * 4);
    }
    TR_TRY(st->tiles.ensure(o));
    char *b = st->tiles.as<char>();
    GeomStats *gs = (GeomStats *)(b + o_gs);
    CParam *cp = (CParam *)(b + o_cp);
    unsigned *cell = (unsigned *)(b + o_cell);
    double *mat = (double *)(b + o_mat);
    int4 *geo = (int4 *)(b + o_geo);
    float4 *recA = (float4 *)(b + o_A), *recB = (float4 *)(b + o_B);
    p.gs = gs;
    p.cp = cp;
    p.cell = cell;
    p.mat = mat;
    p.geo = geo;
    p.recA = recA;
    p.recB = recB;
    p.nodes = (double *)(b + o_nodes);
    const unsigned lb = (unsigned)std::max<size_t>(1, std::min<size_t>((n + 255) / 256, 152 * 16));

    if (a.timing) TR_TRY(cudaEventRecord(a.ev_begin, s));
    if (a.timing && a.ev_main0) TR_TRY(cudaEventRecord(a.ev_main0, s));
    for (int pass = 0; pass < nc_all; pass += nc_pass) {
        const CondDev *conds = a.conds_dev + pass;
        p.sigma = a.sigma + (size_t)pass * (size_t)a.grid.n;
        p.L = a.L;
        unsigned *gmax = nullptr;
        k_tree_prep<<<1, 32, 0, s>>>(conds, nc_pass, gs);
        if (a.L.n_broad > 0) {
            gmax = (unsigned *)(b + o_gmax);
            TR_TRY(cudaMemsetAsync(gmax, 0, (size_t)nc_pass * 4, s));
            TR_TRY(launch_line_gamma(a.L, n, conds, nc_pass, (float *)(b + o_glc), gmax, s));
            p.L.gamma_lc = (float *)(b + o_glc);
            p.L.gamma_stride = nc_pass;
            *launches += 1;
        }
        k_tree_geom<<<lb, 256, 0, s>>>(a.L, n, a.grid.nu_A, a.grid.step, a.grid.n, a.opts.cutoff,
                                       per_cond ? a.opts.width_mult : 0.0, conds, zero_k, 1.5, geo, gs);
        if (a.opts.threshold != XC_THRESHOLD_NONE) {
            const int words = (nc_pass + 31) / 32;
            uint32_t *keep = (uint32_t *)(b + o_keep);
            TR_TRY(launch_line_keep(a.L, n, conds, nc_pass, strength_sel(a.opts), keep, words, s));
            p.L.keep = keep;
            p.L.keep_words = words;
            *launches += 1;
        }
        const int setup = 1 + (p.ncell + 1 + (p.far ? TR_MAT : 0) + 255) / 256;
        k_tree_setup<<<setup, 256, 0, s>>>(p, conds, nc_pass, cp, a.opts.quantity, gmax, cell, mat);
        *launches += 3;
        for (int c0 = 0; c0 < nc_pass; c0 += cg) {
            const int m = std::min(cg, nc_pass - c0);
            p.c0 = c0;
            p.n_cond = m;
            (ext ? fn.rec_ext : fn.rec)<<<dim3(lb, m), 256, 0, s>>>(p, recA, recB);
            *launches += 2;
            if (p.far) {
                const int64_t tasks = (int64_t)p.nblk[0] + p.nblk[1] + p.nblk[2];
                p.wpt = warps_per_task(tasks * m);
                const int per = TR_W / p.wpt;
                fn.nodes<<<dim3((unsigned)((tasks + per - 1) / per), m), TR_T, 0, s>>>(p);
                *launches += 1;
            }
            const int64_t tasks = ((int64_t)p.n_pts + 31) / 32;
            p.wpt = warps_per_task(tasks * m);
            const int per = TR_W / p.wpt;
            fn.points<<<dim3((unsigned)((tasks + per - 1) / per), m), TR_T, 0, s>>>(p);
        }
    }
    if (a.timing && a.ev_main1) TR_TRY(cudaEventRecord(a.ev_main1, s));
    if (a.timing && a.ev_core1) TR_TRY(cudaEventRecord(a.ev_core1, s));
    if (a.timing) TR_TRY(cudaEventRecord(a.ev_end, s));
    TR_TRY(cudaGetLastError());
    char lbuf[160];
    snprintf(lbuf, sizeof(lbuf), "profile %d: block-interpolated sweep, %d conditions per pass", a.opts.profile, cg);
    st->last_tuning = lbuf;
    return XC_OK;
}

}  // namespace xc
