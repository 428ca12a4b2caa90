// xc_tree64.cu -- the plain FP64 cross section with the far field interpolated on blocks.
//
// The scheme of xc_tree.cu (see there for the taking rule and the poles) in FP64 throughout:
// blocks of 512 and 128 points with 32 Chebyshev nodes.  A block takes a line from a gap of
// 0.47 B, where the degree-31 interpolant of 1/(x - s)^2 is within 1e-16 of every value.
// What bounds it is the FP64 pipe (2 lanes per cycle and SM on GB300, 1/64 of FP32), so the
// count of FP64 operations is all that matters and integer work beside them is free:
//   * a 2500-step cut costs ~450 nodes and ~330 points per line instead of 5000 points;
//   * region I of w4 is its real rational in u = D^2 (6 operations), four lines to a
//     reciprocal at the nodes, instead of the complex quotient (~55);
//   * regions III and IV, a few points per line, are numbered line after line and evaluated 32
//     at a time: a branch taken by one lane costs the FP64 pipe as much as by 32.
// 1e5 lines on 200 001 points: 46.2 ms for the direct sum (59 FP64 operations per pair).
//
// Sums are formed so that they do not depend on where the scanned chunks of lines begin
// (line order within each sum, groups of four counted from the block's first line), and
// blocks are aligned to multiples of the grid step, so that a shard of the grid with an exact
// step gives the same bits as the whole.  Nodes are kept as unevaluated sums of two doubles,
// and the interpolation at a point includes the first-order term of the rounding of its
// wavenumber nu_A + k step, so neither adds to the rounding of the direct sum.
#include <math.h>

#include <algorithm>

#include "xc_internal.cuh"
#include "xc_once.h"
#include "xc_profile64.cuh"
#include "xc_tree.cuh"

namespace xc {

constexpr int T64_M = 32;
__device__ __host__ constexpr int t64_block(int lev) { return lev == 0 ? 128 : 512; }
__device__ __host__ constexpr int t64_gap(int lev) { return lev == 0 ? 60 : 240; }
constexpr int T64_MAT_UP = 0;                                   // [4][32 source][32]: 512 -> 128
constexpr int T64_MAT_PT = 4 * T64_M * T64_M;                   // [32 source][128]: 128 -> points
constexpr int T64_MAT_DV = T64_MAT_PT + T64_M * 128;            // its derivative, per grid step
constexpr int T64_MAT = T64_MAT_DV + T64_M * 128;

struct T64Params {
    TreeParams t;                 // geo: x = n, y..z = cut range (not clipped to the grid)
    const double *nu, *I, *al, *ga;
    int *count;                   // lines taken by each block, level 1 first
    float acoef;                  // alpha / nu, rounded up
    int koff;                     // blocks start at multiples of their size minus koff
};

// Bringing the node sums to a point costs 96 FP64 operations whatever the list.  Points whose blocks
// took no more than this many lines evaluate them instead (a value takes about 15 operations with
// the plain Lorentzian and w4's quads, 60 with the binned Lorentzian's arctangent, 20 times that for the
// Gauss-Hermite sums).  A line that a block takes covers all its points, so every shard of the grid that
// holds one of them counts the same lines.  1e6 points, 3000 lines, cut 50 and 256 steps, us, direct sum /
// nodes always / so: Lorentz 95 / 310 / 106 and 128 / 334 / 141, w4 186 / 422 / 215 and 295 / 463 / 271,
// binned Gauss-Hermite Voigt 932 / 1135 / 908 and 3203 / 3091 / 2835.
template <int PROF>
constexpr int t64_few() {
    return PROF == XC_LORENTZ || PROF == XC_VOIGT_W4 ? 6 : (PROF == XC_LORENTZ_BINNED ? 1 : 0);
}
// whether the points of the 128-point block j (parent j / 4) use its nodes
template <int PROF>
__device__ __forceinline__ bool t64_far(const T64Params &q, int j) {
    return q.t.far && q.count[j >> 2] + q.count[q.t.nblk[1] + j] > t64_few<PROF>();
}

__device__ __forceinline__ double t64_node(int B, int m) {
    return (double)(rintf(64.f * (float)(B - 1) * (1.f - cospif((float)(2 * m + 1) * (1.f / (2 * T64_M))))) * (1.f / 128.f));
}

// Lagrange basis polynomial of node m at x (grid steps from the first point of a block of B
// points with nodes xn)
__device__ double t64_basis(const double *xn, int B, int m, double x) {
    const double xm = xn[m], s = 4.0 / (double)B;
    double num = 1.0, den = 1.0;
#pragma unroll 4
    for (int j = 0; j < T64_M; ++j) {
        const double f = j == m ? 1.0 : (x - xn[j]) * s, g = j == m ? 1.0 : (xm - xn[j]) * s;
        num *= f;
        den *= g;
    }
    return num / den;
}

// per line: integer grid position and the range of indices inside the cut (any integers);
// zero_k > 0: profiles that are exactly 0 in FP64 beyond zero_k alpha
__global__ void __launch_bounds__(256) k_t64_geom(const double *__restrict__ nu, const double *__restrict__ al,
                                                  const double *__restrict__ cut, size_t n, double nu_A, double step,
                                                  double zero_k, int4 *geo) {
    const double inv_h = 1.0 / step;
    for (size_t l = (size_t)blockIdx.x * 256 + threadIdx.x; l < n; l += (size_t)gridDim.x * 256) {
        const double v = nu[l];
        double c = cut[l];
        const double pos = floor((v - nu_A) * inv_h);
        int4 g = make_int4((int)fmin(fmax(pos, kPosMin), kPosMax), 1, 0, 0);
        // grids of fewer than 2^30 points and cuts of fewer than 2^20 steps: a line beyond the clamp
        // reaches no point.  A negative cut: left out by the intensity threshold.
        if (c >= 0.0 && pos > kPosMin && pos < kPosMax) {
            if (zero_k > 0.0) c = fmin(c, zero_k * al[l] + 2.0 * step);
            int64_t ka = (int64_t)ceil((v - c - nu_A) * inv_h), kb = (int64_t)floor((v + c - nu_A) * inv_h);
            while (__dsub_rn(grid_x(nu_A, step, ka - 1), v) >= -c) --ka;
            while (__dsub_rn(grid_x(nu_A, step, ka), v) < -c) ++ka;
            while (__dsub_rn(grid_x(nu_A, step, kb + 1), v) <= c) ++kb;
            while (__dsub_rn(grid_x(nu_A, step, kb), v) > c) --kb;
            if (ka <= kb) {
                g.y = (int)i64max(ka, -0x7fffffff);
                g.z = (int)i64min(kb, 0x7fffffff);
            }
        }
        geo[l] = g;
    }
}

__global__ void __launch_bounds__(64) k_t64_setup(TreeParams p, unsigned *cell) {
    const int i = blockIdx.x * 64 + threadIdx.x;
    if (i > p.ncell) return;
    const int v = p.cell0 + TR_CELL * i;
    size_t a = 0, b = p.n;
    while (a < b) {
        const size_t m = a + ((b - a) >> 1);
        if (p.geo[m].x < v) a = m + 1; else b = m;
    }
    cell[i] = (unsigned)a;
}

__global__ void __launch_bounds__(64) k_t64_mat(double *mat) {
    __shared__ double xn[2][T64_M];   // nodes of a 128- and a 512-point block
    xn[threadIdx.x / T64_M][threadIdx.x % T64_M] = t64_node(t64_block(threadIdx.x / T64_M), threadIdx.x % T64_M);
    __syncthreads();
    const int k = blockIdx.x * 64 + threadIdx.x;
    if (k >= T64_MAT_DV) return;
    if (k < T64_MAT_PT) {
        const int j = k / (T64_M * T64_M), s = (k / T64_M) % T64_M, d = k % T64_M;
        mat[k] = t64_basis(xn[1], 512, s, (double)(128 * j) + xn[0][d]);
    } else {
        const int q = k - T64_MAT_PT, s = q / 128;
        const double x = (double)(q % 128);
        mat[k] = t64_basis(xn[0], 128, s, x);
        // the derivative multiplies a rounding error: three digits of it are plenty
        mat[k + (T64_MAT_DV - T64_MAT_PT)] = (t64_basis(xn[0], 128, s, x + 1e-3) - t64_basis(xn[0], 128, s, x - 1e-3)) * 500.0;
    }
}

// the handle's interpolation matrices (constants), made by its first call that needs them
cudaError_t tree64_mat(DevBuf *buf, cudaStream_t s) {
    return make_once(*buf, (size_t)T64_MAT * sizeof(double), [&] {
        k_t64_mat<<<(T64_MAT_DV + 63) / 64, 64, 0, s>>>(buf->as<double>());
        return cudaGetLastError();
    });
}

// w4 region I in u = D^2: I V = P (u + C) / (u^2 + E u + C^2), with s = alpha^2 / ln 2,
// Y = ln 2 gamma^2 / alpha^2, C = s (Y + 1/2), E = 2 s (Y - 1/2)
struct W4Line {
    double nu, E, F, P, PC, ia, y, amp;
};
__device__ __forceinline__ W4Line t64_line(const T64Params &p, size_t l) {
    W4Line w;
    const double al = p.al[l];
    w.nu = p.nu[l];
    w.ia = kSqrtLn2 / al;
    w.y = p.ga[l] * w.ia;
    w.amp = p.I[l] * (0.46971863934982566 / kSqrtLn2) * w.ia;
    const double s = al * al * (1.0 / kLn2), Y = w.y * w.y, C = s * (Y + 0.5);
    w.E = 2.0 * s * (Y - 0.5);
    w.F = C * C;
    w.P = w.amp * 0.5641896 * w.y * s;
    w.PC = w.P * C;
    return w;
}

// ---------------------------------------------------------------------------
// nodes: a warp owns a block, a lane a node
// ---------------------------------------------------------------------------
constexpr int T64_RING = 36;   // accepted lines held: up to 3 left over and 32 new ones

// Two warps per CTA and the large blocks first: an SM's FP64 pipe is the limit, so the blocks
// (a 512-point one has five times the lines of a 128-point one) are spread in small pieces.
constexpr int T64_NW = 2;
template <int PROF>
__global__ void __launch_bounds__(32 * T64_NW) k_t64_nodes(T64Params q) {
    constexpr bool W4 = PROF == XC_VOIGT_W4;
    __shared__ double sL[T64_NW][T64_RING * (W4 ? 5 : 4)];
    __shared__ double sX[64], sW[64];
    const TreeParams &p = q.t;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (p.ngh > 0) {
        if (threadIdx.x < p.ngh) {
            sX[threadIdx.x] = p.ghx[threadIdx.x];
            sW[threadIdx.x] = p.ghw[threadIdx.x];
        }
        __syncthreads();
    }
    int task = blockIdx.x * T64_NW + warp;
    const int lev = task < p.nblk[1] ? 1 : 0;
    if (lev == 0) task -= p.nblk[1];
    if (task >= p.nblk[lev]) return;
    const int B = t64_block(lev), b0 = task * B - q.koff, b1 = b0 + B - 1;
    if (b1 < 0 || b0 >= p.n_pts) return;   // outside the grid (alignment): nothing reads its nodes
    const float ac = q.acoef;
    const int D = tr_radius(p, ac, t64_gap(lev), b1);
    const bool up = lev == 0;
    const int p0 = (task & ~3) * 128 - q.koff, p1 = p0 + 511;   // the parent of a 128-point block
    const int Dp = up ? tr_radius(p, ac, t64_gap(1), p1) : 0;
    const Segs sg = tr_far_segs(p, b0, b1, D, up, p0, p1, Dp);
    // the node's wavenumber as an unevaluated sum xh + xl
    const double t = (double)b0 + t64_node(B, lane);
    const double pr = __dmul_rn(t, p.step), pe = fma(t, p.step, -pr);
    const double xh = __dadd_rn(p.nu_A, pr), bb = __dsub_rn(xh, p.nu_A);
    const double xl = __dadd_rn(__dadd_rn(__dsub_rn(p.nu_A, __dsub_rn(xh, bb)), __dsub_rn(pr, bb)), pe);
    double *buf = sL[warp];
    double acc = 0.0;
    int held = 0, taken = 0;
    // lines 0..cnt-1 of the buffer, four to a reciprocal; the last ones (only at the end) singly
    auto quad = [&](int j) {
        double Dn[4], N[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const double *w = buf + 5 * (j + i);
            const double d = (xh - w[0]) + xl, u = d * d;
            Dn[i] = fma(u, u + w[1], w[2]);
            N[i] = fma(w[3], u, w[4]);
        }
        const double D01 = Dn[0] * Dn[1], D23 = Dn[2] * Dn[3];
        const double N01 = fma(N[0], Dn[1], N[1] * Dn[0]), N23 = fma(N[2], Dn[3], N[3] * Dn[2]);
        acc = fma(fma(N01, D23, N23 * D01), rcp64(D01 * D23), acc);
    };
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {
        const unsigned e = sg.e[k];
        unsigned i = sg.s[k];
        int4 g = make_int4(0, 1, 0, 0);
        if (i + lane < e) g = p.geo[i + lane];
#pragma unroll 1
        for (; i < e; i += 32u) {
            const unsigned l = i + lane;
            int4 gn = make_int4(0, 1, 0, 0);
            if (l + 32u < e) gn = p.geo[l + 32u];
            const bool ok = l < e && tr_takes(g, b0, b1, b1, D) && !(up && tr_takes(g, p0, p1, p1, Dp));
            const unsigned m = __ballot_sync(0xffffffffu, ok);
            if (m) {
                const int slot = held + __popc(m & ((1u << lane) - 1u));
                if (ok) {
                    if (W4) {
                        const W4Line w = t64_line(q, l);
                        double *b = buf + 5 * slot;
                        b[0] = w.nu;
                        b[1] = w.E;
                        b[2] = w.F;
                        b[3] = w.P;
                        b[4] = w.PC;
                    } else {
                        double *b = buf + 4 * slot;
                        b[0] = q.nu[l];
                        b[1] = q.I[l];
                        b[2] = q.al[l];
                        b[3] = q.ga[l];
                    }
                }
                held += __popc(m);
                taken += __popc(m);
                __syncwarp();
                if (W4) {
                    int j = 0;
                    for (; j + 4 <= held; j += 4) quad(j);
                    // the lines left over move to the front
                    const int rest = held - j;
                    double keep = 0.0;
                    if (lane < 5 * rest) keep = buf[5 * j + lane];
                    __syncwarp();
                    if (lane < 5 * rest) buf[lane] = keep;
                    held = rest;
                } else {
                    for (int j = 0; j < held; ++j) {
                        const double *b = buf + 4 * j;
                        acc += b[1] * profile64<PROF>((xh - b[0]) + xl, p.step, b[2], b[3], sX, sW, p.ngh);
                    }
                    held = 0;
                }
                __syncwarp();
            }
            g = gn;
        }
    }
    for (int j = 0; W4 && j < held; ++j) {
        const double *w = buf + 5 * j;
        const double d = (xh - w[0]) + xl, u = d * d;
        acc = fma(fma(w[3], u, w[4]), rcp64(fma(u, u + w[1], w[2])), acc);
    }
    p.nodes[p.node_off[lev] + task * T64_M + lane] = acc;
    if (lane == 0) q.count[(lev ? 0 : p.nblk[1]) + task] = taken;
}

// ---------------------------------------------------------------------------
// points
// ---------------------------------------------------------------------------
// the interpolated far field at point k = s0 + lane added to v, and the output.  j: the
// 128-point block, o: the point's place in it.
__device__ __forceinline__ void t64_finish(const T64Params &q, bool far, int j, int o, int k, int lane, double v) {
    const TreeParams &p = q.t;
    if (far) {
        const double *up = p.nodes + p.node_off[1] + (j >> 2) * T64_M;
        const double *w = p.mat + T64_MAT_UP + (j & 3) * (T64_M * T64_M) + lane;
        double f = p.nodes[p.node_off[0] + j * T64_M + lane];
#pragma unroll 4
        for (int s = 0; s < T64_M; ++s) f = fma(w[s * T64_M], up[s], f);
        // the point's wavenumber is xk = nu_A + k step as rounded: its distance from the exact one
        const double kd = (double)k, pr = __dmul_rn(kd, p.step), pe = fma(kd, p.step, -pr);
        const double xk = __dadd_rn(p.nu_A, pr), bb = __dsub_rn(xk, p.nu_A);
        const double e = __dadd_rn(__dadd_rn(__dsub_rn(p.nu_A, __dsub_rn(xk, bb)), __dsub_rn(pr, bb)), pe);
        const double *wp = p.mat + T64_MAT_PT + o, *wd = p.mat + T64_MAT_DV + o;
        double a = 0.0, b = 0.0;
#pragma unroll 4
        for (int s = 0; s < T64_M; ++s) {
            const double fs = __shfl_sync(0xffffffffu, f, s);
            a = fma(wp[s * 128], fs, a);
            b = fma(wd[s * 128], fs, b);
        }
        v += fma(b, -e * (double)p.inv_h, a);
    }
    if (k >= 0 && k < p.n_pts) p.sigma[k] = v;
}

// Small CTAs: a value of the binned Gauss-Hermite sum holds a warp for 10 us of its SM's FP64 pipe, so the
// warps of one crowded stretch of the grid go to several SMs
constexpr int T64_PW = 2;
template <int PROF>
__global__ void __launch_bounds__(32 * T64_PW) k_t64_points(T64Params q) {
    __shared__ double sL[T64_PW][32 * 4];
    __shared__ int2 sR[T64_PW][32];
    __shared__ double sX[64], sW[64];
    const TreeParams &p = q.t;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (p.ngh > 0) {
        if (threadIdx.x < p.ngh) {
            sX[threadIdx.x] = p.ghx[threadIdx.x];
            sW[threadIdx.x] = p.ghw[threadIdx.x];
        }
        __syncthreads();
    }
    const int task = blockIdx.x * T64_PW + warp;
    const int s0 = task * 32 - q.koff, s1 = s0 + 31;
    if (s0 >= p.n_pts || s1 < 0) return;
    const int p0 = (task >> 2) * 128 - q.koff, p1 = p0 + 127;
    const bool far = t64_far<PROF>(q, task >> 2);
    const int Dp = far ? tr_radius(p, q.acoef, t64_gap(0), p1) : 0;
    const Segs sg = tr_point_segs(p, far, s0, s1, p0, p1, Dp);
    const double xk = grid_x(p.nu_A, p.step, s0 + lane);
    double *buf = sL[warp];
    double acc = 0.0;
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
        const unsigned e = sg.e[k];
#pragma unroll 1
        for (unsigned i = sg.s[k]; i < e; i += 32u) {
            const unsigned l = i + lane;
            int4 g = make_int4(0, 1, 0, 0);
            if (l < e) g = p.geo[l];
            const bool ok = g.y <= s1 && g.z >= s0 && g.y <= g.z && !(far && tr_takes(g, p0, p1, p1, Dp));
            const unsigned m = __ballot_sync(0xffffffffu, ok);
            if (!m) continue;
            if (ok) {
                const int slot = __popc(m & ((1u << lane) - 1u));
                double *b = buf + 4 * slot;
                b[0] = q.nu[l];
                b[1] = q.I[l];
                b[2] = q.al[l];
                b[3] = q.ga[l];
                sR[warp][slot] = make_int2(g.y - s0, g.z - s0);
            }
            __syncwarp();
            const int cnt = __popc(m);
            for (int j = 0; j < cnt; ++j) {
                const double *b = buf + 4 * j;
                const int2 r = sR[warp][j];
                if (lane >= r.x && lane <= r.y)
                    acc += b[1] * profile64<PROF>(__dsub_rn(xk, b[0]), p.step, b[2], b[3], sX, sW, p.ngh);
            }
            __syncwarp();
        }
    }
    t64_finish(q, far, task >> 2, (task & 3) * 32 + lane, s0 + lane, lane, acc);
}

// Re w in w4's region II, real form (see w4_region2_re)
__device__ __forceinline__ double t64_region2(double X, double y, double Y) {
    constexpr double a = 1.410474, b = 0.5641896, s6 = 2.449489742783178098;
    constexpr double Q1 = (3.0 - s6) / 2.0, Q2 = (3.0 + s6) / 2.0;
    constexpr double A1 = (a - b * Q1) / s6, A2 = -(a - b * Q2) / s6;
    const double Z = X + Y, t1 = Z - Q1, t2 = Z - Q2;
    const double D1 = fma(t1, t1, 4.0 * Q1 * Y), D2 = fma(t2, t2, 4.0 * Q2 * Y);
    const double N1 = A1 * (Z + Q1), N2 = A2 * (Z + Q2);
    return y * fma(N1, D2, N2 * D1) * rcp64(D1 * D2);
}

// region III: real coefficients, so two operations each by division through (z - t)(z - conj t)
__device__ __forceinline__ double t64_region3(double x, double y) {
    const double r = y + y, s = fma(x, x, y * y);
    const double n3 = fma(0.5642236, r, 3.778987);
    const double n2 = fma(r, n3, fma(-s, 0.5642236, 11.96482));
    const double n1 = fma(r, n2, fma(-s, n3, 20.20933));
    const double d4 = r + 6.699398;
    const double d3 = fma(r, d4, 21.69274 - s);
    const double d2 = fma(r, d3, fma(-s, d4, 39.27121));
    const double d1 = fma(r, d2, fma(-s, d3, 38.82363));
    const double Nr = fma(y, n1, fma(-s, n2, 16.4955)), Dr = fma(y, d1, fma(-s, d2, 16.4955));
    const double Ni = x * n1, Di = x * d1;
    return fma(Nr, Dr, Ni * Di) * rcp64(fma(Dr, Dr, Di * Di));
}

// region IV, real part only (no sine)
__device__ __forceinline__ double t64_region4(double x, double y) {
    typedef Cx<double> Z;
    const double ur = (y - x) * (y + x), ui = -2.0 * x * y;
    const Z m = cx<double>(-ur, -ui);
    const Z N = 36183.31 + m * (3321.9905 + m * (1540.787 + m * (219.0313 + m * (35.76683 + m * (1.320522 + 0.56419 * m)))));
    const Z D = 32066.6 + m * (24322.84 + m * (9022.228 + m * (2186.181 + m * (364.2191 + m * (61.57037 +
                m * (1.841439 + m))))));
    const double d = rcp64(D.re * D.re + D.im * D.im);
    const double rr = (N.re * D.re + N.im * D.im) * d, ri = (N.im * D.re - N.re * D.im) * d;
    return exp64(ur) * cos(ui) - (y * rr + x * ri);   // t = y - i x
}

struct W4Buf64 {
    double F[T64_RING * 5]; // lines in region I at all the warp's points, inside the cut: nu, E, F, P, PC
    double Z[32 * 8];       // lines whose zone |x| + y < 15 or an end of whose cut lies there: ..., a, y, amplitude
    unsigned m12[32];       // ... their points in regions I and II
    double I[2][32 * 4];    // lines with items of region III / IV: nu, a, y, amplitude
    int4 R[2][32];          // first item, first point, points of the left run, first point of the right run
    int cnt[2][32];
};

// w4.  Lines that cover the warp's points in region I go four to a reciprocal (8.5 FP64 operations
// a value, against 11 one by one), lines with a zone or an end of their cut there one by one, items of regions III and IV
// as in xc_tree.cu.  One sum for each, in line order; groups of four are counted from the
// warp's first line.  Only lines near the points are classified in FP64.
__global__ void __launch_bounds__(128) k_t64_points_w4(T64Params q) {
    __shared__ W4Buf64 sBuf[4];
    const TreeParams &p = q.t;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int task = blockIdx.x * 4 + warp;
    const int s0 = task * 32 - q.koff, s1 = s0 + 31;
    if (s0 >= p.n_pts || s1 < 0) return;
    const int p0 = (task >> 2) * 128 - q.koff, p1 = p0 + 127;
    const int Dp = tr_radius(p, q.acoef, t64_gap(0), p1);
    const int core = tr_radius(p, q.acoef, -(1 << 28), p1) + 1;   // the zones' radius alone
    const bool far = t64_far<XC_VOIGT_W4>(q, task >> 2);
    const Segs sg = tr_point_segs(p, far, s0, s1, p0, p1, Dp);
    const double xk = grid_x(p.nu_A, p.step, s0 + lane), x0 = grid_x(p.nu_A, p.step, s0);
    const double inv_h = 1.0 / p.step;
    const unsigned below = (1u << lane) - 1u;
    W4Buf64 &buf = sBuf[warp];
    double accF = 0.0, accZ = 0.0, acc34[2] = {0.0, 0.0};
    int held = 0;
    // the numerator and denominator of region I of list line j at this lane's point
    auto one = [&](int j, double &N, double &Dn) {
        const double *w = buf.F + 5 * j;
        const double d = __dsub_rn(xk, w[0]), u = d * d;
        Dn = fma(u, u + w[1], w[2]);
        N = fma(w[3], u, w[4]);
    };
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
        const unsigned e = sg.e[k];
#pragma unroll 1
        for (unsigned i = sg.s[k]; i < e; i += 32u) {
            const unsigned l = i + lane;
            int4 g = make_int4(0, 1, 0, 0);
            if (l < e) g = p.geo[l];
            const bool ok = g.y <= s1 && g.z >= s0 && g.y <= g.z && !(far && tr_takes(g, p0, p1, p1, Dp));
            if (!__any_sync(0xffffffffu, ok)) continue;
            W4Line w{};
            bool zone = false;
            unsigned cut = 0u, m3 = 0u, m34 = 0u;
            int k0 = 0, k1 = -1, k30 = 0, k31 = -1;
            if (ok) {
                w = t64_line(q, l);
                const int ka = max(g.y - s0, 0), kb = min(g.z - s0, 31);
                cut = lanes_of(ka, kb);
                if (g.x >= s0 - core && g.x <= s1 + core && w.y < 15.0) {
                    const double pos = (w.nu - x0) * inv_h, ra = q.al[l] * (1.0 / kSqrtLn2) * inv_h;   // 1/a in grid steps
                    const double rz = (15.0 - w.y) * ra + 1e-3;
                    zone = pos + rz >= 0.0 && pos - rz <= 31.0;
                    if (zone && w.y < 5.5) {
                        const double r34 = (5.5 - w.y) * ra, r3 = fmin(r34, (w.y + 0.176) * (1.0 / 0.195) * ra);
                        k0 = max((int)ceil(fmax(pos - r34, -1.0)), ka);
                        k1 = min((int)floor(fmin(pos + r34, 32.0)), kb);
                        k30 = max((int)ceil(fmax(pos - r3, -1.0)), k0);
                        k31 = min((int)floor(fmin(pos + r3, 32.0)), k1);
                        m34 = lanes_of(k0, k1);
                        m3 = lanes_of(k30, k31);
                    }
                }
            }
            const unsigned m4 = m34 & ~m3, m12 = cut & ~m34;
            // groups of four only of lines that cover all 32 points: a grid shard, which holds the lines
            // that reach its own points, then forms the same groups
            const bool isF = ok && !zone && cut == 0xffffffffu, isZ = ok && !isF && m12 != 0u;
            const unsigned bF = __ballot_sync(0xffffffffu, isF), bZ = __ballot_sync(0xffffffffu, isZ);
            const unsigned b34[2] = {__ballot_sync(0xffffffffu, m3 != 0u), __ballot_sync(0xffffffffu, m4 != 0u)};
            if (isF) {
                const int slot = held + __popc(bF & below);
                double *b = buf.F + 5 * slot;
                b[0] = w.nu;
                b[1] = w.E;
                b[2] = w.F;
                b[3] = w.P;
                b[4] = w.PC;
            }
            held += __popc(bF);
            if (isZ) {
                const int slot = __popc(bZ & below);
                double *b = buf.Z + 8 * slot;
                b[0] = w.nu;
                b[1] = w.E;
                b[2] = w.F;
                b[3] = w.P;
                b[4] = w.PC;
                b[5] = w.ia;
                b[6] = w.y;
                b[7] = w.amp;
                buf.m12[slot] = m12;
            }
            int tot[2];
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const unsigned m = t == 0 ? m3 : m4;
                tot[t] = 0;
                if (b34[t] == 0u) continue;
                const int ni = __popc(m);
                int off = ni;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(0xffffffffu, off, o);
                    if (lane >= o) off += v;
                }
                tot[t] = __shfl_sync(0xffffffffu, off, 31);
                if (ni > 0) {
                    const int slot = __popc(b34[t] & below);
                    double *b = buf.I[t] + 4 * slot;
                    b[0] = w.nu;
                    b[1] = w.ia;
                    b[2] = w.y;
                    b[3] = w.amp;
                    const int left = t == 1 && m3 != 0u ? k30 - k0 : ni;
                    buf.R[t][slot] = make_int4(off - ni, t == 0 ? k30 : k0, left, k31 + 1);
                    buf.cnt[t][slot] = ni;
                }
            }
            __syncwarp();
            int j4 = 0;
            for (; j4 + 4 <= held; j4 += 4) {
                double N[4], Dn[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) one(j4 + j, N[j], Dn[j]);
                const double D01 = Dn[0] * Dn[1], D23 = Dn[2] * Dn[3];
                const double N01 = fma(N[0], Dn[1], N[1] * Dn[0]), N23 = fma(N[2], Dn[3], N[3] * Dn[2]);
                accF = fma(fma(N01, D23, N23 * D01), rcp64(D01 * D23), accF);
            }
            if (j4) {   // the lines left over move to the front
                const int rest = held - j4;
                double keep = 0.0;
                if (lane < 5 * rest) keep = buf.F[5 * j4 + lane];
                __syncwarp();
                if (lane < 5 * rest) buf.F[lane] = keep;
                held = rest;
            }
            const int nZ = __popc(bZ);
            for (int j = 0; j < nZ; ++j) {
                const double *b = buf.Z + 8 * j;
                const bool in = (buf.m12[j] >> lane) & 1u;
                const double d = __dsub_rn(xk, b[0]), u = d * d;
                const double x = fabs(d) * b[5], y = b[6];
                const bool first = x + y >= 15.0;
                double v = 0.0;
                if (__any_sync(0xffffffffu, in && !first)) v = b[7] * t64_region2(x * x, y, y * y);
                if (__any_sync(0xffffffffu, in && first)) {
                    const double v1 = fma(b[3], u, b[4]) * rcp64(fma(u, u + b[1], b[2]));
                    v = first ? v1 : v;
                }
                if (in) accZ += v;
            }
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                int line0 = 0;
                for (int b = 0; b < tot[t]; b += 32) {
                    int first = -1;
                    if (lane < __popc(b34[t])) first = buf.R[t][lane].x - b;
                    const unsigned starts = __reduce_or_sync(0xffffffffu, first >= 0 && first < 32 ? 1u << first : 0u);
                    const int line = line0 + __popc(starts & (below | (1u << lane))) - 1;
                    double v = 0.0;
                    if (b + lane < tot[t]) {
                        const double *w4 = buf.I[t] + 4 * line;
                        const int4 r = buf.R[t][line];
                        const int o = b + lane - r.x;
                        const int kp = o < r.z ? r.y + o : r.w + o - r.z;
                        const double x = fabs(__dsub_rn(grid_x(p.nu_A, p.step, s0 + kp), w4[0])) * w4[1];
                        v = w4[3] * (t == 0 ? t64_region3(x, w4[2]) : t64_region4(x, w4[2]));
                    }
                    const int jl = __shfl_sync(0xffffffffu, line, min(31, tot[t] - 1 - b));
                    for (int j = __shfl_sync(0xffffffffu, line, 0); j <= jl; ++j) {
                        const int4 r = buf.R[t][j];
                        int o = lane - r.y;
                        if (o >= r.z) o = lane - r.w >= 0 ? lane - r.w + r.z : -1;
                        const int it = r.x + o - b;
                        const double a = __shfl_sync(0xffffffffu, v, it & 31);
                        if (o >= 0 && o < buf.cnt[t][j] && it >= 0 && it < 32) acc34[t] += a;
                    }
                    line0 += __popc(starts);
                }
            }
            __syncwarp();
        }
    }
    for (int j = 0; j < held; ++j) {
        double N, Dn;
        one(j, N, Dn);
        accF = fma(N, rcp64(Dn), accF);
    }
    t64_finish(q, far, task >> 2, (task & 3) * 32 + lane, s0 + lane, lane, (accF + accZ) + (acc34[0] + acc34[1]));
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
// bytes of scratch behind the int4 geometry of n lines
static size_t tree64_layout(const xc_grid &g, double cutoff, size_t n, TreeParams *p, size_t *o_cell, size_t *o_nodes,
                            size_t *o_count) {
    p->n = n;
    p->n_pts = (int)g.n;
    p->nu_A = g.nu_A;
    p->step = g.step;
    p->cutoff = cutoff;
    p->inv_h = (float)(1.0 / g.step);
    p->reach = (int)ceil(cutoff / g.step) + 2;
    p->cell0 = -TR_CELL * ((p->reach + 2 * TR_CELL) / TR_CELL);
    p->ncell = (int)(((int64_t)p->n_pts - p->cell0 + p->reach + 2 * TR_CELL) / TR_CELL);
    int off = 0;
    for (int lev = 1; lev >= 0; --lev) {
        p->nblk[lev] = (p->n_pts + 511 + t64_block(lev) - 1) / t64_block(lev);   // any alignment
        p->node_off[lev] = off;
        off += p->nblk[lev] * T64_M;
    }
    p->nblk[2] = 0;
    size_t o = 0;
    auto carve = [&](size_t bytes) { size_t r = o; o += (bytes + 255) & ~size_t(255); return r; };
    carve(n * sizeof(int4));
    *o_cell = carve((size_t)(p->ncell + 1) * 4);
    *o_nodes = carve((size_t)off * 8);
    *o_count = carve((size_t)(p->nblk[0] + p->nblk[1]) * 4);
    return o;
}

size_t tree64_scratch(const xc_grid &g, double cutoff, size_t n) {
    TreeParams p;
    size_t a, b, c;
    return tree64_layout(g, cutoff, n, &p, &a, &b, &c);
}

template <int PROF>
static void t64_launch(const T64Params &q, int64_t *launches, cudaStream_t s) {
    if (q.t.far) {
        k_t64_nodes<PROF><<<(q.t.nblk[0] + q.t.nblk[1] + T64_NW - 1) / T64_NW, 32 * T64_NW, 0, s>>>(q);
        *launches += 1;
    }
    const int64_t tasks = ((int64_t)q.t.n_pts + q.koff + 31) / 32;
    if (PROF == XC_VOIGT_W4)
        k_t64_points_w4<<<(unsigned)((tasks + 3) / 4), 128, 0, s>>>(q);
    else
        k_t64_points<PROF><<<(unsigned)((tasks + T64_PW - 1) / T64_PW), 32 * T64_PW, 0, s>>>(q);
    *launches += 1;
}

cudaError_t launch_tree64(int profile, const double *nu, const double *I, const double *al, const double *ga,
                          const double *cut, size_t n, double acoef, const xc_grid &g, double cutoff, bool fixed_cut,
                          const double *ghx, const double *ghw, int ngh, const double *mat, void *scratch,
                          double *sigma, int64_t *launches, cudaStream_t s) {
    T64Params q;
    TreeParams &p = q.t;
    size_t o_cell, o_nodes, o_count;
    tree64_layout(g, cutoff, n, &p, &o_cell, &o_nodes, &o_count);
    char *b = static_cast<char *>(scratch);
    int4 *geo = reinterpret_cast<int4 *>(b);
    unsigned *cell = reinterpret_cast<unsigned *>(b + o_cell);
    p.geo = geo;
    p.cell = cell;
    p.mat = mat;
    p.nodes = reinterpret_cast<double *>(b + o_nodes);
    q.count = reinterpret_cast<int *>(b + o_count);
    p.sigma = sigma;
    p.ghx = ghx;
    p.ghw = ghw;
    p.ngh = 0;
    p.wpt = 1;
    const bool dop = profile == XC_DOPPLER || profile == XC_DOPPLER_BINNED;
    const bool w4 = profile == XC_VOIGT_W4;
    p.far = dop ? 0 : 1;
    p.cover = fixed_cut && !dop ? std::max(0, (int)floor(cutoff / g.step) - 2) : 0;
    p.core = w4 ? 18.05f : 0.f;
    p.ext = 0.f;
    p.ext0 = 1;
    if (w4) {
        p.ext = 0.86f;
        p.ext0 = 2;
    } else if (profile == XC_LORENTZ_BINNED) {
        p.ext0 = 2;
    } else if (profile == XC_VOIGT_GH_BINNED || profile == XC_VOIGT_GH_SAMPLED) {
        p.ngh = ngh;
        p.ext = (float)(sqrt(2.0 * ngh + 2.0) / 0.83255) * 1.001f;
        p.ext0 = 3;
    }
    q.nu = nu;
    q.I = I;
    q.al = al;
    q.ga = ga;
    const double a0 = nearbyint(g.nu_A / g.step);
    q.koff = fabs(a0) < 1e15 ? (int)(((int64_t)a0 % 512 + 512) % 512) : 0;
    q.acoef = (float)(acoef * (1.0 + 1e-6));
    const unsigned lb = (unsigned)std::max<size_t>(1, std::min<size_t>((n + 255) / 256, 152 * 16));
    // exp(-x) and erfc(x) are exactly 0 in FP64 from x = 745.2 and x = 27.3 on: 32.8 alpha for both
    k_t64_geom<<<lb, 256, 0, s>>>(nu, al, cut, n, g.nu_A, g.step, dop ? 33.2 : 0.0, geo);
    k_t64_setup<<<(unsigned)((p.ncell + 1 + 63) / 64), 64, 0, s>>>(p, cell);
    *launches += 2;
    switch (profile) {
    case XC_DOPPLER: t64_launch<XC_DOPPLER>(q, launches, s); break;
    case XC_LORENTZ: t64_launch<XC_LORENTZ>(q, launches, s); break;
    case XC_VOIGT_W4: t64_launch<XC_VOIGT_W4>(q, launches, s); break;
    case XC_VOIGT_GH_BINNED: t64_launch<XC_VOIGT_GH_BINNED>(q, launches, s); break;
    case XC_VOIGT_GH_SAMPLED: t64_launch<XC_VOIGT_GH_SAMPLED>(q, launches, s); break;
    case XC_DOPPLER_BINNED: t64_launch<XC_DOPPLER_BINNED>(q, launches, s); break;
    case XC_LORENTZ_BINNED: t64_launch<XC_LORENTZ_BINNED>(q, launches, s); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace xc
