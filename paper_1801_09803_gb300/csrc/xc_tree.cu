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
#include "xc_once.h"
#include "xc_tree.cuh"

namespace xc {

constexpr int TR_FOLD = 4;                  // scanned chunks (32 lines) per FP32 partial sum at the nodes
                                            // (each chunk at the points, where one strong line can
                                            // dominate: 512 lines in one sum left 6e-7 of rounding)
// the largest alpha / nu of conditions c0 .. c0 + n - 1 of the pass
__device__ __forceinline__ float tr_group_acoef(const TreeParams &p, int c0, int n) {
    float a = 0.f;
    for (int c = 0; c < n; ++c) a = fmaxf(a, p.cp[p.c0 + c0 + c].acoef);
    return a;
}

template <int PROF>
__device__ __forceinline__ float tr_amplitude(const float4 &A) {
    return (PROF == XC_VOIGT_W4 || PROF == XC_VOIGT_GH_SAMPLED || PROF == XC_LORENTZ_BINNED) ? A.z
           : PROF == XC_VOIGT_GH_BINNED                                                     ? A.w
                                                                                            : A.y;
}
template <int PROF>
constexpr bool tr_pairs() { return PROF == XC_VOIGT_W4 || PROF == XC_LORENTZ; }

// w4's region II (see w4_region2_re) of two lines: X = x^2, Y = y^2, yP = y times the amplitude
__device__ __forceinline__ f32x2 w4_region2_pair(f32x2 X, f32x2 Y, f32x2 yP) {
    constexpr double a = 1.410474, b = 0.5641896, s6 = 2.449489742783178098;
    constexpr float Q1 = (float)((3.0 - s6) / 2.0), Q2 = (float)((3.0 + s6) / 2.0);
    constexpr float A1 = (float)((a - b * ((3.0 - s6) / 2.0)) / s6);
    constexpr float A2 = (float)(-(a - b * ((3.0 + s6) / 2.0)) / s6);
    const f32x2 Z = add2(X, Y);
    const f32x2 t1 = add2(Z, pk2(-Q1, -Q1)), t2 = add2(Z, pk2(-Q2, -Q2));
    const f32x2 D1 = fma2(t1, t1, mul2(Y, pk2(4.f * Q1, 4.f * Q1)));
    const f32x2 D2 = fma2(t2, t2, mul2(Y, pk2(4.f * Q2, 4.f * Q2)));
    const f32x2 N1 = mul2(pk2(A1, A1), add2(Z, pk2(Q1, Q1))), N2 = mul2(pk2(A2, A2), add2(Z, pk2(Q2, Q2)));
    return mul2(mul2(yP, fma2(N1, D2, mul2(N2, D1))), rcp2(mul2(D1, D2)));
}

__device__ __forceinline__ float sum2(f32x2 v) {
    float a, b;
    upk2(v, a, b);
    return a + b;
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
// Line geometry in grid steps and the intensity statistics.  width_mult > 0: the cut of
// condition *cond; zero_k > 0: profiles that are exactly 0 in FP32 beyond zero_k nu + zero_0
// (cm^-1) of the centre, for the largest alpha of the conditions.
// Bound by the FP64 pipe.  The estimates of the range's ends are exact unless they lie within
// eps of an integer (eps: many times their rounding error); only then the exact predicate
// settles them (57 -> about 25 FP64 operations per line; 0.91 -> 0.60 ms for 1e7 lines).
__global__ void __launch_bounds__(256) k_tree_geom(LinesDev L, size_t n, double nu_A, double step, int64_t n_pts,
                                                   double cutoff, double width_mult, const CondDev *cond,
                                                   double zero_k, double zero_0, double eps, double inv_h,
                                                   int4 *geo, GeomStats *gs) {
    float m1 = 0.f, m2 = 0.f;
    double ac = 0.0, lnTr = 0.0, gsc = 0.0;
    CondDev c{};
    if (width_mult > 0.0) {
        c = *cond;
        ac = alpha_coef(c.T, c.mass_da);
        lnTr = log(c.T_ref / c.T);
        gsc = c.P / c.P_ref;
    }
    for (size_t l = (size_t)blockIdx.x * 256 + threadIdx.x; l < n; l += (size_t)gridDim.x * 256) {
        const double nu = L.nu[l];
        const float gr = L.gamma_ref[l], nT = L.n_T[l];
        double cut = cutoff;
        if (width_mult > 0.0) {
            const double ga = L.n_broad > 0 ? mixture_gamma64(L, l, c.n_shift, lnTr, c.gamma_scale * gsc)
                                            : c.gamma_scale * f2d(gr) * exp64((f2d(nT) + c.n_shift) * lnTr) * gsc;
            cut = fmin(width_mult * fmax(ac * nu, ga), cutoff);
        }
        if (zero_k > 0.0) cut = fmin(cut, zero_k * nu + zero_0);
        const double d = (nu - nu_A) * inv_h;
        const double fl = floor(d);
        const double flc = fmin(fmax(fl, kPosMin), kPosMax);
        const double ta = (nu - cut - nu_A) * inv_h, tb = (nu + cut - nu_A) * inv_h;
        int ka = 1, kb = 0;
        if (fabs(ta - rint(ta)) > eps && fabs(tb - rint(tb)) > eps) {
            const double top = (double)n_pts;   // < 2^30
            if (ta <= top && tb >= -1.0) {
                ka = max(0, (int)ceil(fmax(ta, -1.0)));
                kb = (int)floor(fmin(tb, top - 1.0));
            }
        } else {
            int64_t k0, k1;
            line_k_range(nu, cut, nu_A, step, inv_h, n_pts, &k0, &k1);
            ka = (int)i64min(i64max(k0, -1), (int64_t)0x7fffffff);
            kb = (int)i64min(i64max(k1, -1), (int64_t)0x7fffffff);
        }
        if (kb < ka) { ka = 1; kb = 0; }
        geo[l] = make_int4((int)flc, ka, kb, __float_as_int((float)(d - fl)));
        const float gA = (float)L.g_up[l] * L.A[l];
        const float nuf = (float)nu;
        m1 = fmaxf(m1, gA / (nuf * nuf));
        m2 = fmaxf(m2, gA / nuf);
    }
    // two atomics per CTA: one per warp and statistic on the same words took longer than the lines
    __shared__ float sm[2][8];
    m1 = isfinite(m1) ? m1 : 0.f;
    m2 = isfinite(m2) ? m2 : 0.f;
    for (int o = 16; o > 0; o >>= 1) {
        m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, o));
        m2 = fmaxf(m2, __shfl_xor_sync(0xffffffffu, m2, o));
    }
    if ((threadIdx.x & 31) == 0) {
        sm[0][threadIdx.x >> 5] = m1;
        sm[1][threadIdx.x >> 5] = m2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) {
            m1 = fmaxf(m1, sm[0][w]);
            m2 = fmaxf(m2, sm[1][w]);
        }
        atomicMax(&gs->gA_nu2_bits, __float_as_uint(m1));   // non-negative floats: integer order
        atomicMax(&gs->gA_nu_bits, __float_as_uint(m2));
        if (blockIdx.x == 0) gs->nu_bits = __float_as_uint(__double2float_ru(L.nu[n - 1]));   // sorted
    }
}

// Lagrange basis polynomial of node m at x, from the block's nodes xn as rounded
__device__ double tr_basis(const float *xn, int B, int m, double x) {
    const double xm = (double)xn[m], s = 4.0 / (double)B;   // scaled: the products stay near 1
    double num = 1.0, den = 1.0;
#pragma unroll
    for (int j = 0; j < TR_M; ++j) {
        const double xj = (double)xn[j];
        num *= j == m ? 1.0 : (x - xj) * s;
        den *= j == m ? 1.0 : (xm - xj) * s;
    }
    return num / den;
}

// entry k of the interpolation matrices; xn: the nodes of each level
__device__ double tr_mat_entry(int k, const float (*xn)[TR_M]) {
    if (k < TR_MAT_128) {
        const int j = k / (TR_M * TR_M), s = (k / TR_M) % TR_M, d = k % TR_M;
        return tr_basis(xn[2], 512, s, (double)(64 * j) + (double)xn[0][d]);
    }
    if (k < TR_MAT_PT) {
        const int q = k - TR_MAT_128, j = q / (TR_M * TR_M), s = (q / TR_M) % TR_M, d = q % TR_M;
        return tr_basis(xn[1], 128, s, (double)(64 * j) + (double)xn[0][d]);
    }
    const int q = k - TR_MAT_PT;
    return tr_basis(xn[0], 64, q / 64, (double)(q % 64));
}

// block 0: per-condition constants, a field (or two) per warp so that their FP64 chains run side
// by side; block 1..: line index
__global__ void __launch_bounds__(128) k_tree_setup(TreeParams p, const CondDev *conds, int n_cond, CParam *cp,
                                                    int quantity, unsigned *cell) {
    if (blockIdx.x == 0) {
        // conditions in order of alpha / nu (as T / mass): those taken together have similar zones
        __shared__ float key[1024];
        const bool order = n_cond > 1 && n_cond <= 1024;
        if (order) {
            for (int c = threadIdx.x; c < n_cond; c += 128) key[c] = (float)conds[c].T / (float)conds[c].mass_da;
            __syncthreads();
        }
        for (int c = threadIdx.x & 31; c < n_cond; c += 32) {
            const CondDev d = conds[c];
            int r = c;
            if (order) {
                r = 0;
                for (int j = 0; j < n_cond; ++j) r += key[j] < key[c] || (key[j] == key[c] && j < c);
            }
            switch (threadIdx.x >> 5) {
            case 0: cparam_strength(d, p.gs, quantity, &cp[r]); break;
            case 1: cparam_temperature(d, &cp[r]); break;
            case 2: cparam_widths(d, &cp[r]); break;
            default:
                cp[r].log2Tr = (float)log2(d.T_ref / d.T);
                cp[r].row = c;
                cp[r].vv_split = 4.f;
                cp[r].vv_beta = 0;
                cp[r].dbound = 0.f;
            }
        }
        return;
    }
    const int i = (blockIdx.x - 1) * 128 + threadIdx.x;
    if (i <= p.ncell) {
        const int v = p.cell0 + TR_CELL * i;
        size_t a = 0, b = p.n;
        while (a < b) {
            const size_t m = a + ((b - a) >> 1);
            if (p.geo[m].x < v) a = m + 1; else b = m;
        }
        cell[i] = (unsigned)a;
    }
}

__global__ void __launch_bounds__(128) k_tree_mat(double *mat) {
    __shared__ float xn[TR_LEVELS][TR_M];
    if (threadIdx.x < TR_LEVELS * TR_M)
        xn[threadIdx.x / TR_M][threadIdx.x % TR_M] = tr_node(tr_block(threadIdx.x / TR_M), threadIdx.x % TR_M);
    __syncthreads();
    const int k = blockIdx.x * 128 + threadIdx.x;
    if (k < TR_MAT) mat[k] = tr_mat_entry(k, xn);
}

static double geom_eps(const xc_grid &g, double cutoff) {
    // 64 times the rounding of a line's position in grid steps
    return std::max(1e-9, 64.0 * 2.3e-16 * (fabs(g.nu_A) + g.step * (double)g.n + 2.0 * cutoff) / g.step);
}

cudaError_t launch_fp32_setup(const LinesDev &L, size_t n, const CondDev *conds, int nc, const xc_grid &grid,
                              double cutoff, int4 *geo, GeomStats *gs, CParam *cp, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(gs, 0, sizeof(GeomStats), s);
    if (e != cudaSuccess) return e;
    if (n)
        k_tree_geom<<<(unsigned)std::min<size_t>((n + 255) / 256, 152 * 8), 256, 0, s>>>(
            L, n, grid.nu_A, grid.step, grid.n, cutoff, 0.0, nullptr, 0.0, 0.0, geom_eps(grid, cutoff), 1.0 / grid.step,
            geo, gs);
    TreeParams p{};
    p.gs = gs;
    p.ncell = -1;
    if (nc) k_tree_setup<<<1, 128, 0, s>>>(p, conds, nc, cp, XC_ABSORPTION, nullptr);
    return cudaGetLastError();
}

// the handle's interpolation matrices (constants), made by its first call that needs them
cudaError_t tree_mat(BatchedState *st, const double **mat, cudaStream_t s) {
    const cudaError_t e = make_once(st->tree_mat, TR_MAT * sizeof(double),
                                    [&] { return launch_tree_mat(st->tree_mat.as<double>(), s); });
    *mat = st->tree_mat.as<double>();
    return e;
}

cudaError_t launch_tree_mat(double *mat, cudaStream_t s) {
    k_tree_mat<<<(TR_MAT + 127) / 128, 128, 0, s>>>(mat);
    return cudaGetLastError();
}

// profile constants of the group's conditions, for the lines that can reach the grid (a contiguous range of
// the sorted list: 32 conditions of a 301-point Lorentz window in 1e7 lines 2.55 ms with all lines', 0.69 so)
template <int PROF, bool EXT>
__global__ void __launch_bounds__(256) k_tree_recs(TreeParams p, float4 *recA, float4 *recB) {
    const int c = blockIdx.y;
    const CParam cp = p.cp[p.c0 + c];
    const float h = (float)p.step;
    const size_t l1 = tr_upper(p, p.n_pts + p.reach + 1);
    const size_t l0 = tr_lower(p, -p.reach) & ~63u;   // whole sectors for a warp
    for (size_t l = l0 + (size_t)blockIdx.x * 256 + threadIdx.x; l < l1; l += (size_t)gridDim.x * 256) {
        float4 A, B = make_float4(0.f, 0.f, 0.f, -1.f), S;
        float t2;
        line_consts<PROF, EXT>(p.L, l, cp, h, p.inv_h, &A, &B, &t2, &S);
        recA[(size_t)c * p.n + l] = A;
        if (PROF == XC_VOIGT_W4) recB[(size_t)c * p.n + l] = B;
    }
}

// ---------------------------------------------------------------------------
// far levels: sums at the nodes.  A lane holds two of the block's 16 nodes, and the four
// quarter-warps take different lines (one node and two half-warps for the profiles that are
// costly per value: fewer lines to fill an iteration).  Per 32 scanned lines the accepted ones are compacted
// into shared memory, pairs of lines interleaved for the packed arithmetic; one iteration
// takes 8 lines.  (With one node per lane and two line streams the loop was bound by the
// shared-memory reads: 81 % of their rate at the 1e7-line list on 2e6 points, 1.65 ms.)
// ---------------------------------------------------------------------------
template <int PROF>
__global__ void __launch_bounds__(TR_T) k_tree_nodes(TreeParams p) {
    constexpr int PAIR = tr_pairs<PROF>() ? (PROF == XC_VOIGT_W4 ? 3 : 2) : 2;   // 16-byte words per pair
    __shared__ float4 sL[TR_W][tr_pairs<PROF>() ? 16 * PAIR : 48];   // non-pairs: 24 bytes a line
    __shared__ float sX[64], sW[64];
    __shared__ double sRed[TR_W][TR_M];
    constexpr int R = tr_pairs<PROF>() ? 2 : 1, LN = TR_M / R, NS = 32 / LN;   // nodes per lane, lanes per stream, streams
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, strm = lane / LN;
    if (p.ngh > 0) {
        if (threadIdx.x < p.ngh) {
            sX[threadIdx.x] = (float)p.ghx[threadIdx.x];
            sW[threadIdx.x] = (float)p.ghw[threadIdx.x];
        }
        __syncthreads();
    }
    // Neighbouring tasks share a CTA: they read the same lines (dealt out over the CTAs instead,
    // the 32-condition table took 27 ms more).  The large blocks have the most lines, so each
    // level has its own number of warps per task.
    int lev = 2, cta = blockIdx.x;
    while (lev > 0 && cta >= p.ncta[lev]) cta -= p.ncta[lev--];
    const int wpt = p.wptl[lev], part = warp % wpt;
    const int task = cta * (TR_W / wpt) + warp / wpt;
    const int c = blockIdx.y;
    const bool live = task < p.nblk[lev];
    float hi[2] = {0.f, 0.f}, lo[2] = {0.f, 0.f};
    if (live) {
        const float ac = p.cp[p.c0 + c].acoef;
        const int B = tr_block(lev), b0 = task * B, b1 = b0 + B - 1, b1c = min(b1, p.n_pts - 1);
        const int D = tr_radius(p, ac, tr_gap(lev), b1);
        const bool up = lev < 2;
        const int PB = up ? tr_block(lev + 1) : 1;
        const int p0 = up ? b0 / PB * PB : 0, p1 = p0 + PB - 1, p1c = min(p1, p.n_pts - 1);
        const int Dp = up ? tr_radius(p, ac, tr_gap(lev + 1), p1) : 0;
        const Segs sg = tr_far_segs(p, b0, b1, D, up, p0, p1, Dp);
        const float x[2] = {tr_node(B, R * (lane % LN)), tr_node(B, R * (lane % LN) + R - 1)};
        const f32x2 xa = pk2(x[0], x[0]), xb = pk2(x[1], x[1]);
        const float4 *recA = p.recA + (size_t)c * p.n;
        float4 *buf = sL[warp];
        f32x2 acca = 0ull, accb = 0ull;
        float acc[2] = {0.f, 0.f};
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
                    constexpr int pad = tr_pairs<PROF>() ? 2 * NS : NS;
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
                        for (int j = strm; 2 * j < cnt; j += NS) {
                            const ulonglong2 *q = reinterpret_cast<const ulonglong2 *>(buf + j * PAIR);
                            const ulonglong2 nf = q[0], c0 = q[1];
                            ulonglong2 c1 = c0;
                            if (PROF == XC_VOIGT_W4) c1 = q[2];
                            const f32x2 da = sub2(sub2(xa, nf.x), nf.y), db = sub2(sub2(xb, nf.x), nf.y);
                            const f32x2 ua = mul2(da, da), ub = mul2(db, db);
                            if (PROF == XC_VOIGT_W4) {
                                acca = fma2(fma2(c1.x, ua, c1.y), rcp2(fma2(ua, add2(ua, c0.x), c0.y)), acca);
                                accb = fma2(fma2(c1.x, ub, c1.y), rcp2(fma2(ub, add2(ub, c0.x), c0.y)), accb);
                            } else {
                                acca = fma2(c0.y, rcp2(add2(ua, c0.x)), acca);
                                accb = fma2(c0.y, rcp2(add2(ub, c0.x)), accb);
                            }
                        }
                    } else {
                        // binned Gauss-Hermite: the short arctangent when all the chunk's lines allow it
                        const bool far = PROF == XC_VOIGT_GH_BINNED &&
                                         __all_sync(0xffffffffu, !ok || gh_far(A.y, (float)D, A.x * p.gh_ext));
                        for (int j = strm; j < cnt; j += NS) {
                            const float2 *q = reinterpret_cast<const float2 *>(buf) + j * 3;
                            const float2 nf = q[0], a01 = q[1], a23 = q[2];
                            const float4 Ac = make_float4(a01.x, a01.y, a23.x, a23.y);
#pragma unroll
                            for (int r = 0; r < R; ++r) {
                                const float d = (x[r] - nf.x) - nf.y;
                                acc[r] += far ? gh_far_value(d, Ac, sX, sW, p.ngh)
                                              : contrib_single<PROF>(d * d, d, Ac, make_float4(0.f, 0.f, 0.f, -1.f), sX, sW,
                                                                     p.ngh);
                            }
                        }
                    }
                    __syncwarp();
                    if (++in_fold == TR_FOLD) {
                        if (tr_pairs<PROF>()) {
                            acc[0] = sum2(acca);
                            acc[1] = sum2(accb);
                            acca = accb = 0ull;
                        }
                        tr_fold(hi[0], lo[0], acc[0]);
                        tr_fold(hi[1], lo[1], acc[1]);
                        in_fold = 0;
                    }
                }
                g = gn;
            }
        }
        if (tr_pairs<PROF>()) {
            acc[0] = sum2(acca);
            acc[1] = sum2(accb);
        }
        tr_fold(hi[0], lo[0], acc[0]);
        tr_fold(hi[1], lo[1], acc[1]);
    }
    // the line streams' (and the task's warps') sums, in a fixed order
    double v[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        v[r] = (double)hi[r] + (double)lo[r];
        if (LN == 8) v[r] += __shfl_xor_sync(0xffffffffu, v[r], 8);
        v[r] += __shfl_xor_sync(0xffffffffu, v[r], 16);
    }
    if (wpt > 1) {
        __syncthreads();
        if (lane < LN)
#pragma unroll
            for (int r = 0; r < R; ++r) sRed[warp][R * lane + r] = v[r];
        __syncthreads();
        if (part == 0 && lane < LN)
            for (int w = 1; w < wpt; ++w)
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] += sRed[warp + w][R * lane + r];
    }
    if (live && part == 0 && lane < LN) {
        double *out = p.nodes + (size_t)c * p.nodes_per_cond + p.node_off[lev] + task * TR_M + R * lane;
#pragma unroll
        for (int r = 0; r < R; ++r) out[r] = v[r];
    }
}

// w4 at the nodes, CG (2 or 4) conditions at a time.  A line's position, its range tests, its place in the
// shared-memory list and u = delta^2 are the same for every condition; a condition adds its
// constants and 6 packed instructions per node and pair of lines.  The group's blocks use the
// largest alpha of its conditions (they are ordered by alpha).  32 conditions x 1e7 lines:
// 53 ms one condition at a time, 33 ms four.
template <int CG>
__global__ void __launch_bounds__(TR_T, 3) k_tree_nodes_w4(TreeParams p) {
    constexpr int PAIR = 1 + 2 * CG, NS = 4;   // 16-byte words per pair of lines; line streams
    __shared__ float4 sL[TR_W][16 * PAIR];
    __shared__ double sRed[TR_W][CG][TR_M];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, strm = lane >> 3;
    int lev = 2, cta = blockIdx.x;
    while (lev > 0 && cta >= p.ncta[lev]) cta -= p.ncta[lev--];
    const int wpt = p.wptl[lev], part = warp % wpt;
    const int task = cta * (TR_W / wpt) + warp / wpt;
    const int c0 = blockIdx.y * CG, nc = min(CG, p.n_cond - c0);
    const bool live = task < p.nblk[lev];
    float hi[CG][2], lo[CG][2];
#pragma unroll
    for (int q = 0; q < CG; ++q) hi[q][0] = hi[q][1] = lo[q][0] = lo[q][1] = 0.f;
    if (live) {
        const float ac = tr_group_acoef(p, c0, nc);
        const int B = tr_block(lev), b0 = task * B, b1 = b0 + B - 1, b1c = min(b1, p.n_pts - 1);
        const int D = tr_radius(p, ac, tr_gap(lev), b1);
        const bool up = lev < 2;
        const int PB = up ? tr_block(lev + 1) : 1;
        const int p0 = up ? b0 / PB * PB : 0, p1 = p0 + PB - 1, p1c = min(p1, p.n_pts - 1);
        const int Dp = up ? tr_radius(p, ac, tr_gap(lev + 1), p1) : 0;
        const Segs sg = tr_far_segs(p, b0, b1, D, up, p0, p1, Dp);
        const float xn0 = tr_node(B, 2 * (lane & 7)), xn1 = tr_node(B, 2 * (lane & 7) + 1);
        const f32x2 xa = pk2(xn0, xn0), xb = pk2(xn1, xn1);
        const float4 *recA = p.recA + (size_t)c0 * p.n;
        float4 *buf = sL[warp];
        f32x2 acc[CG][2];
#pragma unroll
        for (int q = 0; q < CG; ++q) acc[q][0] = acc[q][1] = 0ull;
        int in_fold = 0;
        auto fold = [&]() {
#pragma unroll
            for (int q = 0; q < CG; ++q)
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    float a = sum2(acc[q][r]);
                    acc[q][r] = 0ull;
                    tr_fold(hi[q][r], lo[q][r], a);
                }
        };
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
                float4 A[CG];
                bool any = false;
#pragma unroll
                for (int q = 0; q < CG; ++q) {
                    A[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (ok && q < nc) A[q] = recA[(size_t)q * p.n + l];
                    any |= A[q].z != 0.f;
                }
                ok &= any;
                const unsigned m = __ballot_sync(0xffffffffu, ok);
                const int cnt = __popc(m);
                if (cnt) {
                    const unsigned below = (1u << lane) - 1u;
                    int slot = __popc(m & below);
                    float n = (float)(g.x - b0), f = __int_as_float(g.w);
                    bool put = ok;
                    if (!ok) {   // lanes that fill the last iteration with lines of amplitude 0
                        const int z = __popc(~m & below);
                        put = z < ((-cnt) & (2 * NS - 1));
                        slot = cnt + z;
                        n = -1e4f;
                        f = 0.f;
#pragma unroll
                        for (int q = 0; q < CG; ++q) A[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                    if (put) {
                        float *w = reinterpret_cast<float *>(buf) + (slot >> 1) * (4 * PAIR) + (slot & 1);
                        w[0] = n;
                        w[2] = f;
#pragma unroll
                        for (int q = 0; q < CG; ++q) {
                            w[4 + 8 * q] = A[q].x;
                            w[6 + 8 * q] = A[q].y;
                            w[8 + 8 * q] = A[q].z;
                            w[10 + 8 * q] = A[q].w;
                        }
                    }
                    __syncwarp();
                    for (int j = strm; 2 * j < cnt; j += NS) {
                        const ulonglong2 *w = reinterpret_cast<const ulonglong2 *>(buf + j * PAIR);
                        const ulonglong2 nf = w[0];
                        const f32x2 da = sub2(sub2(xa, nf.x), nf.y), db = sub2(sub2(xb, nf.x), nf.y);
                        const f32x2 ua = mul2(da, da), ub = mul2(db, db);
#pragma unroll
                        for (int q = 0; q < CG; ++q) {
                            const ulonglong2 k0 = w[1 + 2 * q], k1 = w[2 + 2 * q];
                            acc[q][0] = fma2(fma2(k1.x, ua, k1.y), rcp2(fma2(ua, add2(ua, k0.x), k0.y)), acc[q][0]);
                            acc[q][1] = fma2(fma2(k1.x, ub, k1.y), rcp2(fma2(ub, add2(ub, k0.x), k0.y)), acc[q][1]);
                        }
                    }
                    __syncwarp();
                    if (++in_fold == TR_FOLD) {
                        fold();
                        in_fold = 0;
                    }
                }
                g = gn;
            }
        }
        fold();
    }
    // the line streams' (and the task's warps') sums, in a fixed order
    double v[CG][2];
#pragma unroll
    for (int q = 0; q < CG; ++q)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            v[q][r] = (double)hi[q][r] + (double)lo[q][r];
            v[q][r] += __shfl_xor_sync(0xffffffffu, v[q][r], 8);
            v[q][r] += __shfl_xor_sync(0xffffffffu, v[q][r], 16);
        }
    if (wpt > 1) {
        __syncthreads();
        if (lane < 8)
#pragma unroll
            for (int q = 0; q < CG; ++q) {
                sRed[warp][q][2 * lane] = v[q][0];
                sRed[warp][q][2 * lane + 1] = v[q][1];
            }
        __syncthreads();
        if (part == 0 && lane < 8)
            for (int w = 1; w < wpt; ++w)
#pragma unroll
                for (int q = 0; q < CG; ++q) {
                    v[q][0] += sRed[warp + w][q][2 * lane];
                    v[q][1] += sRed[warp + w][q][2 * lane + 1];
                }
    }
    if (live && part == 0 && lane < 8)
#pragma unroll
        for (int q = 0; q < CG; ++q)
            if (q < nc)
                reinterpret_cast<double2 *>(p.nodes + (size_t)(c0 + q) * p.nodes_per_cond + p.node_off[lev] +
                                            task * TR_M)[lane] = make_double2(v[q][0], v[q][1]);
}

// ---------------------------------------------------------------------------
// points: the pairs no block takes, plus the interpolated sums.  A warp owns 32 points.
// This kernel takes every profile but w4: Lorentzians in packed pairs of lines, masked by
// the cut, the other profiles one line at a time.
// ---------------------------------------------------------------------------
// the interpolated far field at the warp's 32 points (from s0) added to v, and the output
__device__ __forceinline__ void tr_finish(const TreeParams &p, int c, int s0, int lane, double v) {
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

template <int PROF>
__global__ void __launch_bounds__(TR_T) k_tree_points(TreeParams p) {
    constexpr bool PAIRS = tr_pairs<PROF>();
    __shared__ float4 sL[TR_W][PAIRS ? 16 * 3 : 32 * 2];   // pairs: n, f | cut ranges | constants; singles: n, f, ka, kb | A
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
        const int Dp = p.far ? tr_radius(p, p.cp[p.c0 + c].acoef, tr_gap(0), p1) : 0;
        const Segs sg = tr_point_segs(p, p.far, s0, s1, p0, p1, Dp);
        const float x = (float)lane;
        const f32x2 x2 = pk2(x, x);
        const float4 *recA = p.recA + (size_t)c * p.n;
        float4 *buf = sL[warp];
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
                float4 A = make_float4(0.f, 0.f, 0.f, 0.f);
                if (ok) {
                    A = recA[l];
                    ok = tr_amplitude<PROF>(A) != 0.f;
                }
                const unsigned m = __ballot_sync(0xffffffffu, ok);
                if (m) {
                    const unsigned below = (1u << lane) - 1u;
                    const int cnt = __popc(m);
                    const float n = (float)(g.x - s0), f = __int_as_float(g.w);
                    const int ka = max(g.y - s0, 0), kb = min(g.z - s0, 31);
                    float acc = 0.f;
                    if (PAIRS) {
                        const bool fill = !ok && (cnt & 1) && __popc(~m & below) == 0;   // completes the last pair
                        if (ok || fill) {
                            const int slot = fill ? cnt : __popc(m & below);
                            float *q = reinterpret_cast<float *>(buf) + (slot >> 1) * 12 + (slot & 1);
                            q[0] = fill ? -1e4f : n;
                            q[2] = fill ? 0.f : f;
                            q[4] = __int_as_float(fill ? 0 : ka);
                            q[6] = __int_as_float(fill ? -1 : kb - ka);
                            q[8] = fill ? 0.f : A.x;
                            q[10] = fill ? 0.f : A.y;
                        }
                        __syncwarp();
                        f32x2 acc2 = 0ull;
#pragma unroll 2
                        for (int j = 0; 2 * j < cnt; ++j) {
                            const ulonglong2 *q = reinterpret_cast<const ulonglong2 *>(buf + j * 3);
                            const ulonglong2 nf = q[0], c0 = q[2];
                            const int4 kk = reinterpret_cast<const int4 *>(buf + j * 3)[1];   // ka1 ka2 w1 w2
                            const f32x2 d = sub2(sub2(x2, nf.x), nf.y);
                            float v1, v2;
                            upk2(mul2(c0.y, rcp2(add2(mul2(d, d), c0.x))), v1, v2);
                            v1 = lane - kk.x >= 0 && lane - kk.x <= kk.z ? v1 : 0.f;
                            v2 = lane - kk.y >= 0 && lane - kk.y <= kk.w ? v2 : 0.f;
                            acc2 = add2(acc2, pk2(v1, v2));
                        }
                        acc = sum2(acc2);
                    } else {
                        if (ok) {
                            float4 *q = buf + __popc(m & below) * 2;
                            const bool far = PROF == XC_VOIGT_GH_BINNED &&
                                             gh_far(A.y, (float)max(s0 - g.x, g.x - s1), A.x * p.gh_ext);
                            q[0] = make_float4(n, f, __int_as_float(ka), __int_as_float(far ? kb + 64 : kb));
                            q[1] = A;
                        }
                        __syncwarp();
                        for (int j = 0; j < cnt; ++j) {
                            // a strong line's value in the sum makes the next ones' rounding: 16 a sum
                            if ((j & 15) == 15) tr_fold(hi, lo, acc);
                            const float4 t = buf[2 * j], a = buf[2 * j + 1];
                            const float d = (x - t.x) - t.y;
                            const int ka1 = __float_as_int(t.z), kb1 = __float_as_int(t.w);
                            if (PROF == XC_VOIGT_GH_BINNED && kb1 >= 64) {
                                const float v = gh_far_value(d, a, sX, sW, p.ngh);
                                acc += lane >= ka1 && lane <= kb1 - 64 ? v : 0.f;
                            } else if (lane >= ka1 && lane <= kb1) {
                                acc += contrib_single<PROF>(d * d, d, a, make_float4(0.f, 0.f, 0.f, -1.f), sX, sW, p.ngh);
                            }
                        }
                    }
                    __syncwarp();
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
    if (live && part == 0) tr_finish(p, c, s0, lane, v);
}

// Voigt w4 at the points, CG conditions at a time.  Lines whose zone |x| + y < 15 cannot reach the
// warp's 32 points (most are there for an end of their cut) are in region I at every one of them
// for all conditions: packed pairs of lines, masked by the cut, position and masks shared by the
// conditions.  The lines near the points are then taken condition by condition.  Each lane
// classifies one line, and they go three ways:
//   F  region I at every point of the warp: packed pairs, masked by the cut;
//   Z  the zone reaches the points: packed pairs that evaluate regions I and II and select per
//      point (region I is skipped where no point needs it);
//   items  the points in regions III and IV, which are few per line and costly: numbered line
//      after line, region by region, and evaluated 32 at a time with one region per warp
//      instruction; their owner lanes then add them in line order.
// One line at a time with a branch per region left 22 of 32 lanes active and paid for up to
// four regions per line: 6.4 ms at the 1e7-line list on 2e6 points, 5.5 ms so, 5.1 ms with each
// line's points kept as a bit per lane (an owner's item is the count of the bits below its own;
// from the runs' ends it took a dozen instructions per line).  32 conditions x 1e7 lines: 92 ms
// one condition at a time, 82 ms four, 76 ms with the bits, 73 ms with the odd spacing below.
// Pairs of lines lie an odd number of 16-byte words apart (the last word is not used), so that
// the lanes that write a pair each meet in the same bank two at a time instead of eight.
constexpr int w4_words_f(int nq) { return 3 + 2 * nq; }   // n, f | masks | E, F | P, PC of each condition
constexpr int W4_WORDS_Z = 7;                             // n, f | E, F | P, PC | a^2, y^2 | y Pv, t2 | masks
template <int CG>
struct W4Buf {
    static_assert(w4_words_f(CG) <= w4_words_f(1) + W4_WORDS_Z, "F of all conditions fits");
    // F of CG conditions, or F of one condition followed by Z
    float4 F[16 * (w4_words_f(1) + W4_WORDS_Z)];
    __device__ __forceinline__ float4 *Z() { return F + 16 * w4_words_f(1); }
    float4 I[2][32];               // per line with items of region III / IV: n, f, a, y
    int4 R[2][32];                 // first item, first point, points of the left run, Pv (bits)
    int S[2][32];                  // first point of the right run
    uint2 M[2][32];                // first item, points (a bit per lane)
    float2 sum[CG][32];            // each point's sums (compensated)
};

// inclusive sum over the warp's lanes: the shuffle's own predicate selects the lanes that add
__device__ __forceinline__ unsigned tr_scan(unsigned v) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
        asm volatile(
            "{\n\t.reg .pred p;\n\t.reg .u32 t;\n\t"
            "shfl.sync.up.b32 t|p, %0, %1, 0, 0xffffffff;\n\t"
            "@p add.u32 %0, %0, t;\n\t}"
            : "+r"(v)
            : "r"(o));
    return v;
}

// F pairs of NQ conditions: values at the lane's point (bit: the lane's), masked, into acc
template <int NQ>
__device__ __forceinline__ void w4_masked_pairs(const float4 *F, int nF, unsigned bit, f32x2 x2, float (&acc)[2 * NQ]) {
#pragma unroll 2
    for (int j = 0; 2 * j < nF; ++j) {
        const ulonglong2 *w = reinterpret_cast<const ulonglong2 *>(F + j * w4_words_f(NQ));
        const ulonglong2 nf = w[0];
        const uint2 mk = *reinterpret_cast<const uint2 *>(w + 1);
        const f32x2 d = sub2(sub2(x2, nf.x), nf.y), u = mul2(d, d);
        const bool i1 = (mk.x & bit) != 0u, i2 = (mk.y & bit) != 0u;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const ulonglong2 k0 = w[2 + 2 * q], k1 = w[3 + 2 * q];
            float v1, v2;
            upk2(mul2(fma2(k1.x, u, k1.y), rcp2(fma2(u, add2(u, k0.x), k0.y))), v1, v2);
            if (i1) acc[2 * q] += v1;
            if (i2) acc[2 * q + 1] += v2;
        }
    }
}

template <int CG>
__global__ void __launch_bounds__(CG == 1 ? 256 : 128) k_tree_points_w4(TreeParams p) {
    constexpr int NW = CG == 1 ? 8 : 4;
    __shared__ W4Buf<CG> sBuf[NW];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wpt = p.wpt, part = warp % wpt;
    const int task = blockIdx.x * (NW / wpt) + warp / wpt;
    const int g0 = blockIdx.y * CG, nc = CG == 1 ? 1 : min(CG, p.n_cond - g0);
    const int s0 = task * 32, s1 = s0 + 31;
    const bool live = s0 < p.n_pts;
    W4Buf<CG> &buf = sBuf[warp];
    float2 own = make_float2(0.f, 0.f);   // the sums of a single condition
#pragma unroll
    for (int q = 0; q < CG; ++q) buf.sum[q][lane] = own;
    auto add = [&](int q, float a) {   // the lane's own sums: no other lane touches them
        float2 s = CG == 1 ? own : buf.sum[q][lane];
        tr_fold(s.x, s.y, a);
        if (CG == 1) own = s;
        else buf.sum[q][lane] = s;
    };
    if (live) {
        const int p0 = s0 & ~63, p1 = p0 + 63, p1c = min(p1, p.n_pts - 1);
        const float ac = tr_group_acoef(p, g0, nc);
        const int Dp = tr_radius(p, ac, tr_gap(0), p1);
        const int core = tr_radius(p, ac, -(1 << 28), p1);   // the zones' radius alone
        const Segs sg = tr_point_segs(p, p.far, s0, s1, p0, p1, Dp);
        const float x = (float)lane;
        const f32x2 x2 = pk2(x, x);
        const unsigned below = (1u << lane) - 1u;
        const float4 *recA = p.recA + (size_t)g0 * p.n;
        const float4 *recB = p.recB + (size_t)g0 * p.n;
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
                const bool ok = l < e && g.y <= s1 && g.z >= s0 && g.y <= g.z && !tr_takes(g, p0, p1, p1c, Dp);
                // (a single condition takes all lines in one go)
                const bool near = CG == 1 || (g.x >= s0 - core && g.x <= s1 + core);
                const unsigned bN = __ballot_sync(0xffffffffu, ok && near);
                const unsigned bO = CG == 1 ? 0u : __ballot_sync(0xffffffffu, ok && !near);
                if ((bN | bO) == 0u) {   // most chunks of a width-limited cut
                    g = gn;
                    continue;
                }
                const float n = (float)(g.x - s0), f = __int_as_float(g.w), pos = n + f;
                const int ka = max(g.y - s0, 0), kb = min(g.z - s0, 31);
                const unsigned cut = ok ? lanes_of(ka, kb) : 0u;
                // (distance to the warp's points less a margin)^2: against a zone's radius^2
                const float dist = fmaxf(fmaxf(-pos, pos - 31.f) - 0.1f, 0.f), dist2 = dist * dist;
                if (bO) {
                    const int nF = __popc(bO);
                    if (ok && !near) {
                        const int slot = __popc(bO & below);
                        float *w = reinterpret_cast<float *>(buf.F) + (slot >> 1) * (4 * w4_words_f(CG)) + (slot & 1);
                        w[0] = n;
                        w[2] = f;
                        w[4] = __uint_as_float(cut);
#pragma unroll
                        for (int q = 0; q < CG; ++q) {
                            const float4 A = q < nc ? recA[(size_t)q * p.n + l] : make_float4(0.f, 1.f, 0.f, 0.f);
                            w[8 + 8 * q] = A.x;
                            w[10 + 8 * q] = A.y;
                            w[12 + 8 * q] = A.z;
                            w[14 + 8 * q] = A.w;
                        }
                    }
                    // a pair without a second line: nothing of it is selected
                    if (lane == 0 && (nF & 1))
                        reinterpret_cast<float *>(buf.F)[(nF >> 1) * (4 * w4_words_f(CG)) + 5] = 0.f;
                    __syncwarp();
                    float acc[2 * CG];
#pragma unroll
                    for (int q = 0; q < 2 * CG; ++q) acc[q] = 0.f;
                    w4_masked_pairs<CG>(buf.F, nF, below + 1u, x2, acc);
#pragma unroll
                    for (int q = 0; q < CG; ++q) add(q, acc[2 * q] + acc[2 * q + 1]);
                    __syncwarp();
                }
#pragma unroll 1
                for (int q = 0; bN && q < nc; ++q) {
                    float4 A = make_float4(0.f, 0.f, 0.f, 0.f), B = make_float4(1.f, 1.f, 0.f, -1.f);
                    const bool mine = ok && near;
                    if (mine) {
                        A = recA[(size_t)q * p.n + l];
                        B = recB[(size_t)q * p.n + l];
                    }
                    // zone |x| + y < 15 (with a margin: the points decide by u < t2 themselves)
                    const bool zone = dist2 <= B.w;
                    // points of regions III and IV, |x| + y < 5.5: runs of lanes around the centre
                    unsigned m3 = 0u, m34 = 0u;
                    int k0 = 0, k1 = -1, k30 = 0, k31 = -1;
                    if (zone && B.y < 5.5f && B.z != 0.f) {
                        const float ra = rcp_approx(B.x);
                        const float r34 = (5.5f - B.y) * ra, r3 = fminf(r34, (B.y + 0.176f) * (1.f / 0.195f) * ra);
                        k0 = max(__float2int_ru(fmaxf(pos - r34, -1.f)), ka);
                        k1 = min(__float2int_rd(fminf(pos + r34, 32.f)), kb);
                        k30 = max(__float2int_ru(fmaxf(pos - r3, -1.f)), k0);
                        k31 = min(__float2int_rd(fminf(pos + r3, 32.f)), k1);
                        m34 = lanes_of(k0, k1);
                        m3 = lanes_of(k30, k31);
                    }
                    const unsigned m4 = m34 & ~m3, m12 = cut & ~m34;
                    const bool isZ = zone && m12 != 0u && A.z != 0.f, isF = mine && !zone && A.z != 0.f;
                    const unsigned bF = __ballot_sync(0xffffffffu, isF), bZ = __ballot_sync(0xffffffffu, isZ);
                    const unsigned b3 = __ballot_sync(0xffffffffu, m3 != 0u), b4 = __ballot_sync(0xffffffffu, m4 != 0u);
                    const int nF = __popc(bF), nZ = __popc(bZ);
                    if (isF) {
                        const int slot = __popc(bF & below);
                        float *w = reinterpret_cast<float *>(buf.F) + (slot >> 1) * (4 * w4_words_f(1)) + (slot & 1);
                        w[0] = n;
                        w[2] = f;
                        w[4] = __uint_as_float(cut);
                        w[8] = A.x;
                        w[10] = A.y;
                        w[12] = A.z;
                        w[14] = A.w;
                    }
                    if (isZ) {
                        const int slot = __popc(bZ & below);
                        float *w = reinterpret_cast<float *>(buf.Z()) + (slot >> 1) * (4 * W4_WORDS_Z) + (slot & 1);
                        w[0] = n;
                        w[2] = f;
                        w[4] = A.x;
                        w[6] = A.y;
                        w[8] = A.z;
                        w[10] = A.w;
                        w[12] = B.x * B.x;
                        w[14] = B.y * B.y;
                        w[16] = B.y * B.z;
                        w[18] = B.w;
                        w[20] = __uint_as_float(m12);
                    }
                    if (lane == 0 && (nF & 1)) reinterpret_cast<float *>(buf.F)[(nF >> 1) * (4 * w4_words_f(1)) + 5] = 0.f;
                    if (lane == 1 && (nZ & 1)) reinterpret_cast<float *>(buf.Z())[(nZ >> 1) * (4 * W4_WORDS_Z) + 21] = 0.f;
                    // III (low half) and IV (high half): both counts are summed in one scan
                    unsigned ends = 0u, all = 0u;
                    if ((b3 | b4) != 0u) {
                        ends = tr_scan((unsigned)__popc(m3) | (unsigned)__popc(m4) << 16);
                        all = __shfl_sync(0xffffffffu, ends, 31);
                    }
                    const int tot[2] = {(int)(all & 0xffffu), (int)(all >> 16)};
#pragma unroll
                    for (int t = 0; t < 2; ++t) {
                        const unsigned m = t == 0 ? m3 : m4;
                        if (m != 0u) {
                            const int ni = __popc(m), off = t == 0 ? (int)(ends & 0xffffu) : (int)(ends >> 16);
                            const int slot = __popc((t == 0 ? b3 : b4) & below);
                            buf.I[t][slot] = make_float4(n, f, B.x, B.y);
                            const bool split = t == 1 && m3 != 0u;
                            const int left = t == 0 ? ni : (split ? k30 - k0 : ni);
                            buf.R[t][slot] = make_int4(off - ni, t == 0 ? k30 : k0, left, __float_as_int(B.z));
                            buf.S[t][slot] = k31 + 1;
                            buf.M[t][slot] = make_uint2((unsigned)(off - ni), m);
                        }
                    }
                    __syncwarp();
                    if (nF) {
                        float acc[2] = {0.f, 0.f};
                        w4_masked_pairs<1>(buf.F, nF, below + 1u, x2, acc);
                        add(q, acc[0] + acc[1]);
                    }
                    if (nZ) {
                        float acc1 = 0.f, acc2 = 0.f;
                        for (int j = 0; 2 * j < nZ; ++j) {
                            const ulonglong2 *w = reinterpret_cast<const ulonglong2 *>(buf.Z() + j * W4_WORDS_Z);
                            const ulonglong2 nf = w[0], c0 = w[1], c1 = w[2], ay = w[3], pt = w[4];
                            const uint2 mk = *reinterpret_cast<const uint2 *>(w + 5);
                            const f32x2 d = sub2(sub2(x2, nf.x), nf.y), u = mul2(d, d);
                            float u1, u2, t1, t2, v1, v2;
                            upk2(u, u1, u2);
                            upk2(pt.y, t1, t2);
                            upk2(w4_region2_pair(mul2(u, ay.x), ay.y, pt.x), v1, v2);
                            const bool r1 = u1 >= t1, r2 = u2 >= t2;
                            if (__any_sync(0xffffffffu, r1 || r2)) {
                                float w1, w2;
                                upk2(mul2(fma2(c1.x, u, c1.y), rcp2(fma2(u, add2(u, c0.x), c0.y))), w1, w2);
                                v1 = r1 ? w1 : v1;
                                v2 = r2 ? w2 : v2;
                            }
                            if (mk.x & (below + 1u)) acc1 += v1;
                            if (mk.y & (below + 1u)) acc2 += v2;
                        }
                        add(q, acc1 + acc2);
                    }
#pragma unroll
                    for (int t = 0; t < 2; ++t) {
                        int line0 = 0;                      // lines whose items start before this batch
                        for (int b = 0; b < tot[t]; b += 32) {
                            // lines whose first item lies in this batch: a bit at that item
                            int first = -1;
                            if (lane < __popc(t == 0 ? b3 : b4)) first = (int)buf.M[t][lane].x - b;
                            const unsigned starts =
                                __reduce_or_sync(0xffffffffu, first >= 0 && first < 32 ? 1u << first : 0u);
                            const int line = line0 + __popc(starts & (below | (1u << lane))) - 1;
                            float v = 0.f;
                            if (b + lane < tot[t]) {
                                const float4 w = buf.I[t][line];
                                const int4 r = buf.R[t][line];
                                const int o = b + lane - r.x;
                                const int kp = o < r.z ? r.y + o : buf.S[t][line] + o - r.z;
                                const float xx = w.z * fabsf(((float)kp - w.x) - w.y);
                                v = __int_as_float(r.w) * (t == 0 ? w4_region3_re(xx, w.w) : w4_region4_re(xx, w.w));
                            }
                            // owners add their points' values, line after line
                            const int jl = __shfl_sync(0xffffffffu, line, min(31, tot[t] - 1 - b));
                            float acc = 0.f;
                            for (int j = __shfl_sync(0xffffffffu, line, 0); j <= jl; ++j) {
                                const uint2 r = buf.M[t][j];
                                const int it = (int)r.x + __popc(r.y & below) - b;
                                const float w = __shfl_sync(0xffffffffu, v, it & 31);
                                if ((r.y & (below + 1u)) != 0u && (unsigned)it < 32u) acc += w;
                            }
                            add(q, acc);
                            line0 += __popc(starts);
                        }
                    }
                    __syncwarp();
                }
                g = gn;
            }
        }
    }
    if (CG == 1) buf.sum[0][lane] = own;
    if (wpt > 1) __syncthreads();
    if (!live || part != 0) return;
#pragma unroll 1
    for (int q = 0; q < nc; ++q) {
        double v = 0.0;
        for (int w = 0; w < wpt; ++w) {
            const float2 s = sBuf[warp + w].sum[q][lane];
            v += (double)s.x + (double)s.y;
        }
        tr_finish(p, g0 + q, s0, lane, v);
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
    case XC_VOIGT_W4:
        *f = ProfFns{k_tree_recs<XC_VOIGT_W4, false>, k_tree_recs<XC_VOIGT_W4, true>, nullptr, nullptr};   // see w4_fns
        return true;
    case XC_VOIGT_GH_BINNED: *f = ProfFns TR_FNS(XC_VOIGT_GH_BINNED); return true;
    case XC_VOIGT_GH_SAMPLED: *f = ProfFns TR_FNS(XC_VOIGT_GH_SAMPLED); return true;
    case XC_DOPPLER_BINNED: *f = ProfFns TR_FNS(XC_DOPPLER_BINNED); return true;
    case XC_LORENTZ_BINNED: *f = ProfFns TR_FNS(XC_LORENTZ_BINNED); return true;
    default: return false;
    }
}

// w4's kernels take 1, 2 or 4 conditions at a time
void w4_fns(int cg, ProfFns *f) {
    f->nodes = cg == 4 ? k_tree_nodes_w4<4> : (cg == 2 ? k_tree_nodes_w4<2> : k_tree_nodes<XC_VOIGT_W4>);
    f->points = cg == 4 ? k_tree_points_w4<4> : (cg == 2 ? k_tree_points_w4<2> : k_tree_points_w4<1>);
}

bool is_doppler(int profile) { return profile == XC_DOPPLER || profile == XC_DOPPLER_BINNED; }

// warps per task: several where the tasks alone would leave the SMs with few warps
int warps_per_task(int64_t tasks, int most = TR_W) {
    int w = 1;
    while (w < most && tasks * w < 152 * 16) w *= 2;
    return w;
}

// Profile constants held at a time: 32 conditions of 1e7 lines, eight of 1e8 (four, 12 GB: 1067 ms for 32
// conditions instead of 1041), and no more than half of what the device has free, so that a neighbour
// in the process finds room.
constexpr size_t kMaxRecBytes = (size_t)24 << 30;

}  // namespace

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
    p.gh_ext = 0.f;
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
        p.gh_ext = (float)sqrt(2.0 * a.opts.n_gh + 2.0) * 1.001f;
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

    const size_t rec = n * (w4 ? 32 : 16);
    if ((size_t)cg * rec > std::max(st->tiles.bytes, (size_t)1 << 30)) {   // (the question takes 25 us)
        size_t room = 0, total = 0;
        if (cudaMemGetInfo(&room, &total) != cudaSuccess) cudaGetLastError();
        else cg = (int)std::min<size_t>((size_t)cg, std::max<size_t>(1, (room + st->tiles.bytes) / 2 / rec));
    }
    if (cg < nc_pass && cg > 4) cg &= ~3;   // whole groups of four
    size_t o = 0, o_gs, o_cp, o_cell, o_nodes, o_geo, o_A, o_B, o_keep = 0, o_glc = 0;
    auto carve = [&](size_t bytes) { size_t r = o; o += (bytes + 255) & ~size_t(255); return r; };
    for (;; cg = cg > 4 ? 4 : 1) {
        o = 0;
        o_gs = carve(sizeof(GeomStats));
        o_cp = carve((size_t)nc_pass * sizeof(CParam));
        o_cell = carve((size_t)(p.ncell + 1) * 4);
        o_nodes = carve((size_t)cg * p.nodes_per_cond * 8);
        o_geo = carve(n * sizeof(int4));
        o_A = carve((size_t)cg * n * 16);
        o_B = carve(w4 ? (size_t)cg * n * 16 : 16);
        if (a.opts.threshold != XC_THRESHOLD_NONE) o_keep = carve(n * (size_t)((nc_pass + 31) / 32) * 4);
        if (a.L.n_broad > 0) o_glc = carve(n * (size_t)nc_pass * 4);
        const cudaError_t e = st->tiles.ensure(o);
        if (e == cudaErrorMemoryAllocation && cg > 1) {   // fewer conditions at a time
            cudaGetLastError();
            continue;
        }
        TR_TRY(e);   // out of memory here: the caller falls back to the tiled kernels
        st->tiles_need = o;
        st->tiles_lines = n;
        break;
    }
    char *b = st->tiles.as<char>();
    GeomStats *gs = (GeomStats *)(b + o_gs);
    CParam *cp = (CParam *)(b + o_cp);
    unsigned *cell = (unsigned *)(b + o_cell);
    int4 *geo = (int4 *)(b + o_geo);
    float4 *recA = (float4 *)(b + o_A), *recB = (float4 *)(b + o_B);
    p.gs = gs;
    p.cp = cp;
    p.cell = cell;
    p.mat = nullptr;
    if (p.far) TR_TRY(tree_mat(st, &p.mat, s));
    p.geo = geo;
    p.recA = recA;
    p.recB = recB;
    p.nodes = (double *)(b + o_nodes);
    const unsigned lb = (unsigned)std::max<size_t>(1, std::min<size_t>((n + 255) / 256, 152 * 8));

    const double eps = geom_eps(a.grid, a.opts.cutoff);
    if (a.timing) TR_TRY(cudaEventRecord(a.ev_begin, s));
    if (a.timing && a.ev_main0) TR_TRY(cudaEventRecord(a.ev_main0, s));
    for (int pass = 0; pass < nc_all; pass += nc_pass) {
        const CondDev *conds = a.conds_dev + pass;
        p.sigma = a.sigma + (size_t)pass * (size_t)a.grid.n;
        p.L = a.L;
        TR_TRY(cudaMemsetAsync(gs, 0, sizeof(GeomStats), s));
        if (a.L.n_broad > 0) {
            TR_TRY(launch_line_gamma(a.L, n, conds, nc_pass, (float *)(b + o_glc), nullptr, s));
            p.L.gamma_lc = (float *)(b + o_glc);
            p.L.gamma_stride = nc_pass;
            *launches += 1;
        }
        double am = 0.0;
        for (int c = 0; c < nc_pass; ++c)
            am = std::max(am, alpha_coef(a.conds_host[pass + c].T, a.conds_host[pass + c].mass_da));
        k_tree_geom<<<(unsigned)std::min<size_t>((n + 255) / 256, 152 * 8), 256, 0, s>>>(
            a.L, n, a.grid.nu_A, a.grid.step, a.grid.n, a.opts.cutoff, per_cond ? a.opts.width_mult : 0.0, conds,
            (double)zero_k * am * (1.0 + 1e-6), 1.5 * a.grid.step, eps,
            1.0 / a.grid.step, geo, gs);
        if (a.opts.threshold != XC_THRESHOLD_NONE) {
            const int words = (nc_pass + 31) / 32;
            uint32_t *keep = (uint32_t *)(b + o_keep);
            TR_TRY(launch_line_keep(a.L, n, conds, nc_pass, strength_sel(a.opts), keep, words, s));
            p.L.keep = keep;
            p.L.keep_words = words;
            *launches += 1;
        }
        k_tree_setup<<<1 + (p.ncell + 1 + 127) / 128, 128, 0, s>>>(p, conds, nc_pass, cp, a.opts.quantity, cell);
        *launches += 2;
        for (int c0 = 0; c0 < nc_pass; c0 += cg) {
            const int m = std::min(cg, nc_pass - c0);
            p.c0 = c0;
            p.n_cond = m;
            const int grp = w4 ? (m >= 3 ? 4 : m) : 1, ng = (m + grp - 1) / grp;   // conditions taken together, groups
            if (w4) w4_fns(grp, &fn);
            (ext ? fn.rec_ext : fn.rec)<<<dim3(lb, m), 256, 0, s>>>(p, recA, recB);
            *launches += 2;
            if (p.far) {
                int ctas = 0;
                for (int lev = 0; lev < TR_LEVELS; ++lev) {
                    p.wptl[lev] = warps_per_task((int64_t)p.nblk[lev] * ng);
                    const int per = TR_W / p.wptl[lev];
                    ctas += p.ncta[lev] = (p.nblk[lev] + per - 1) / per;
                }
                fn.nodes<<<dim3((unsigned)ctas, ng), TR_T, 0, s>>>(p);
                *launches += 1;
            }
            const int64_t tasks = ((int64_t)p.n_pts + 31) / 32;
            const int nw = grp == 1 ? TR_W : 4;   // warps per CTA
            p.wpt = warps_per_task(tasks * ng, nw);
            const int per = nw / p.wpt;
            fn.points<<<dim3((unsigned)((tasks + per - 1) / per), ng), 32 * nw, 0, s>>>(p);
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
