// xc_vjp.cu -- adjoint (vector-Jacobian product) of the cross section.
//
// Not in the paper: the chain rule of Eq. (e:int) (intensity), Eq. (e:alphaD),
// Eq. (e:gamma_L) and the profile, applied to sigma_k = sum_l I_l V(nu_k - nu_l;
// alpha_l, gamma_l).  For every line and condition the kernel gathers, over
// the grid points inside the cut,
//     S_I = sum_k g_k V,   S_a = sum_k g_k dV/dalpha,   S_g = sum_k g_k dV/dgamma
// (g = dL/dsigma), recomputing the profile instead of storing it, and then
//     dL/dT_c += I S_I dlnI/dT + I S_a alpha/(2T) - I S_g n gamma/T
//     dL/dP_c += I S_g dgamma/dP,  dL/ds += I S_g dgamma/ds,  dL/dn += I S_g gamma ln(T_ref/T)
//     dL/dgamma_ref_l += I S_g dgamma/dgamma_ref,  dL/dn_l += I S_g gamma ln(T_ref/T)
// with dlnI/dT = c2 E''/T^2 - (c2 nu/T^2)/(exp(c2 nu/T) - 1) - Q'/Q.
//
// Layout: one warp per line (grid-stride), lanes stride over the line's grid
// points, lane c holds the constants of condition c (<= 32 per launch).
// Per-condition scalars are reduced warp -> block in fixed order, written as
// block partials and summed in block order by a second kernel, so the result
// is deterministic.
//
// Two kernels.  k_vjp_lines<PROF> recomputes everything in FP64 (the FP64
// path, and the reference of the finite-difference checks).  k_vjp32<PROF> is the
// FP32 path: GB300 runs FP64 at a small fraction of its FP32 rate, so every
// per-point and per-line quantity is FP32 there and only the per-condition
// accumulators and the per-line outputs are FP64.  It works in grid units
// (delta = k - nu/step, widths a = alpha/step, g = gamma/step) on the line
// geometry and condition constants of the forward FP32 kernels:
//   * w4 region I (the bulk of the points): V = kappa g R, R = (u + C)/((C - u)^2
//     + 4 g^2 u), u = delta^2, b = a^2/(2 ln 2), C = b + g^2, kappa = 0.5641896/sqrt(pi);
//     three sums of g_k times A0 = R, A1 = dR/dC = (1 - 2 (C - u) R')/D with R' = R,
//     and A2 = u R / D (D the denominator), from which
//       sum g V = kappa g S0,   sum g dV/da = kappa g (a/ln 2) S1,
//       sum g dV/dg = kappa (S0 + 2 g^2 (S1 - 4 S2));
//   * regions II-IV (a band around the centre): V = sqrt(ln2/pi)/a Re F,
//     dV/dg = (ln2/sqrt(pi))/a^2 Re F', dV/da = -sqrt(ln2/pi)/a^2 Re(F + t F'), with
//     F + t F' = d(tF)/dt written so that no cancellation is left: its numerator and
//     that of F' expanded once, at compile time, into polynomials whose leading terms
//     cancel exactly in the coefficients (in FP32 the forms
//     F + x dF/dx + y dF/dy and (N'D - ND')/D^2 lose up to 1e-3 of the derivative
//     sums to cancellation in these regions);
//   * per-point FP32 terms are summed in FP32 over 8 points, then into compensated
//     (Kahan) sums; the warp reduction of the sums is compensated too (TwoSum).
#include <math.h>

#include <algorithm>

#include "xc_batched.cuh"
#include "xc_route.h"
#include "xc_tree.cuh"

namespace xc {

constexpr int VT = 256;
constexpr int VW = VT / 32;
constexpr int VMAXC = 32;
constexpr int VMAXB = 8;   // broadeners of a mixture (the limit of xc_set_broadening)

struct VjpLineCond {  // per (line, condition), FP64
    double I, al, ga, dlnI, dga_dP, dga_ds, dga_dgr, lnTr, T;
    double ntga;   // sum over the width's terms of (n + n_shift) gamma: -T dgamma/dT
};

__device__ inline VjpLineCond line_cond64(const LinesDev &L, size_t l, const CondDev &c) {
    VjpLineCond r;
    double nu = L.nu[l];
    double inv_T = 1.0 / c.T;
    double x = kC2 * nu * inv_T;
    double boltz = exp(-kC2 * (double)L.elower[l] * inv_T);
    double stim = -expm1(-x);
    r.I = c.abundance / (8.0 * kPi * kLightCm * c.Q) * (double)L.g_up[l] * (double)L.A[l] / (nu * nu) * boltz * stim;
    r.al = alpha_coef(c.T, c.mass_da) * nu;
    r.lnTr = log(c.T_ref * inv_T);
    double tn = exp(((double)L.n_T[l] + c.n_shift) * r.lnTr);  // (T_ref/T)^n
    double gr = (double)L.gamma_ref[l];
    r.ga = c.gamma_scale * gr * tn * (c.P / c.P_ref);
    r.dga_dP = c.gamma_scale * gr * tn / c.P_ref;
    r.dga_ds = gr * tn * (c.P / c.P_ref);
    r.dga_dgr = c.gamma_scale * tn * (c.P / c.P_ref);
    r.dlnI = kC2 * (double)L.elower[l] * inv_T * inv_T - (x * inv_T) / expm1(x) - c.dQdT / c.Q;
    r.T = c.T;
    r.ntga = ((double)L.n_T[l] + c.n_shift) * r.ga;
    if (L.n_broad > 0) {
        // a mixture of broadeners: gamma = gamma_scale P/P_ref sum_i rho_i gamma_0,i (T_ref/T)^(n_i + n_shift)
        double gu = 0.0, ngu = 0.0;
        for (int i = 0; i < L.n_broad; ++i) {
            const double ni = L.bn[(size_t)i * L.bstride + l] + c.n_shift;
            const double gi = L.bgam[(size_t)i * L.bstride + l] * exp(ni * r.lnTr);
            gu += gi;
            ngu += ni * gi;
        }
        r.ga = c.gamma_scale * gu * (c.P / c.P_ref);
        r.dga_dP = c.gamma_scale * gu / c.P_ref;
        r.dga_ds = gu * (c.P / c.P_ref);
        r.dga_dgr = 0.0;
        r.ntga = c.gamma_scale * ngu * (c.P / c.P_ref);
    }
    return r;
}

__device__ inline double shfl64(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }

// compensated FP32 sum (Kahan): the running compensation keeps the rounding of every
// addition, so the sum is good to a few FP32 ulps of its terms whatever its length
struct KahanF {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float y = __fsub_rn(x, c);
        const float t = __fadd_rn(s, y);
        c = __fsub_rn(__fsub_rn(t, s), y);
        s = t;
    }
    __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

// value and derivatives of the profile (FP64 reference form, all w4 regions)
template <int PROF>
__device__ inline void prof_deriv64(double D, double al, double ga, double *V, double *dVa, double *dVg) {
    if (PROF == XC_DOPPLER) {
        double r = D / al;
        double v = 0.46971863934982566 / al * exp(-kLn2 * r * r);
        *V = v;
        *dVa = v * (-1.0 / al + 2.0 * kLn2 * D * D / (al * al * al));
        *dVg = 0.0;
    } else if (PROF == XC_LORENTZ) {
        double q = D * D + ga * ga;
        *V = ga / (kPi * q);
        *dVa = 0.0;
        *dVg = (D * D - ga * ga) / (kPi * q * q);
    } else {
        double ia = kSqrtLn2 / al;
        Cx<double> dF;
        Cx<double> w = w4_eval<double>(D * ia, ga * ia, &dF);
        double v = 0.46971863934982566 / al * w.re;
        double k2 = kLn2 / (kSqrtPi * al * al);
        double dVD = k2 * dF.im;  // dF/dx = -i F'  ->  Re = Im F'
        double dg = k2 * dF.re;
        *V = v;
        *dVg = dg;
        *dVa = -(v + D * dVD + ga * dg) / al;
    }
}

// Bin average of the Gauss-Hermite Voigt, Eq. (e:sigma:quad), over [D - h/2, D + h/2] and its
// derivatives.  Per node j, s+- = D +- h/2 - alpha x_j/sqrt(ln2), Q+- = s+-^2 + gamma^2:
//   atan(s+/gamma) - atan(s-/gamma) = atan2(gamma h, gamma^2 + s+ s-),
//   d/dgamma = -s+/Q+ + s-/Q- = h (s+ s- - gamma^2)/(Q+ Q-),
//   d/dalpha = (x_j/sqrt(ln2)) gamma (1/Q- - 1/Q+) = (x_j/sqrt(ln2)) gamma h (s+ + s-)/(Q+ Q-),
// the right-hand forms free of the cancellation of the differences in the far wings.
__device__ inline void gh_binned_deriv64(double D, double h, double al, double ga, const double *x, const double *w,
                                         int n, double *V, double *dVa, double *dVg) {
    double v = 0.0, da = 0.0, dg = 0.0;
    const double g2 = ga * ga;
    for (int j = 0; j < n; ++j) {
        const double xs = x[j] / kSqrtLn2;
        const double sp = D + 0.5 * h - al * xs, sm = sp - h;
        // (gamma = 0, a bin's edge exactly on a node: the derivatives have a pole there, taken as 0)
        const double Q = (sp * sp + g2) * (sm * sm + g2), iQ = Q > 0.0 ? 1.0 / Q : 0.0;
        v += w[j] * atan2(ga * h, g2 + sp * sm);
        dg += w[j] * h * (sp * sm - g2) * iQ;
        da += w[j] * xs * ga * h * (sp + sm) * iQ;
    }
    const double k = 1.0 / (kPi * kSqrtPi * h);
    *V = v * k;
    *dVa = da * k;
    *dVg = dg * k;
}

template <int PROF>
__global__ void __launch_bounds__(VT) k_vjp_lines(LinesDev L, size_t n, const CondDev *__restrict__ conds, int nc,
                                                  double nu_A, double step, int64_t n_pts, double cutoff,
                                                  double width_mult, const double *__restrict__ g64,
                                                  double *block_part /*[blk][nc][4 + 2 nb]*/, double *d_gref_line,
                                                  double *d_n_line, int accumulate, const double *ghx,
                                                  const double *ghw, int ngh) {
    __shared__ double s_part[VW][VMAXC][4];
    __shared__ double s_broad[VW][VMAXC][2 * VMAXB];   // mixture: per broadener, scale and n-shift sums
    const int nb = L.n_broad, NQ = 4 + 2 * nb;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double accT = 0.0, accP = 0.0, accS = 0.0, accN = 0.0;  // lane c: condition c
    const CondDev cme = conds[lane < nc ? lane : 0];
    const double inv_step = 1.0 / step;
    for (int q = 0; q < 2 * nb; ++q) s_broad[warp][lane][q] = 0.0;
    for (size_t l = (size_t)blockIdx.x * VW + warp; l < n; l += (size_t)gridDim.x * VW) {
        const double nu = L.nu[l];
        VjpLineCond mine = line_cond64(L, l, cme);
        double line_gr = 0.0, line_n = 0.0;
        int64_t ka0 = 0, kb0 = -1;
        if (!(width_mult > 0.0)) line_k_range(nu, cutoff, nu_A, step, inv_step, n_pts, &ka0, &kb0);
        for (int c = 0; c < nc; ++c) {
            const double I = shfl64(mine.I, c), al = shfl64(mine.al, c), ga = shfl64(mine.ga, c);
            int64_t ka = ka0, kb = kb0;
            if (width_mult > 0.0) line_k_range(nu, fmin(width_mult * fmax(al, ga), cutoff), nu_A, step, inv_step, n_pts, &ka, &kb);
            double SI = 0.0, Sa = 0.0, Sg = 0.0;
            for (int64_t k = ka + lane; k <= kb; k += 32) {
                double D = __dsub_rn(grid_x(nu_A, step, k), nu);
                double V, dVa, dVg;
                if (PROF == XC_VOIGT_GH_BINNED)
                    gh_binned_deriv64(D, step, al, ga, ghx, ghw, ngh, &V, &dVa, &dVg);
                else
                    prof_deriv64<PROF>(D, al, ga, &V, &dVa, &dVg);
                double g = g64[(size_t)c * n_pts + k];
                SI += g * V;
                Sa += g * dVa;
                Sg += g * dVg;
            }
            for (int o = 16; o > 0; o >>= 1) {
                SI += __shfl_xor_sync(0xffffffffu, SI, o);
                Sa += __shfl_xor_sync(0xffffffffu, Sa, o);
                Sg += __shfl_xor_sync(0xffffffffu, Sg, o);
            }
            // every lane holds the sums; lane c owns condition c's scalars
            if (lane == c) {
                const double T = mine.T;
                accT += I * (SI * mine.dlnI + Sa * al / (2.0 * T) - Sg * mine.ntga / T);
                accP += I * Sg * mine.dga_dP;
                accS += I * Sg * mine.dga_ds;
                accN += I * Sg * ga * mine.lnTr;
                // each broadener's term gamma_i: d gamma / d(scale of its gamma_0) = gamma_i,
                // d gamma / d(shift of its n) = gamma_i ln(T_ref/T)
                for (int i = 0; i < nb; ++i) {
                    const double gi = cme.gamma_scale * (cme.P / cme.P_ref) * L.bgam[(size_t)i * L.bstride + l] *
                                      exp((L.bn[(size_t)i * L.bstride + l] + cme.n_shift) * mine.lnTr);
                    s_broad[warp][lane][2 * i] += I * Sg * gi;
                    s_broad[warp][lane][2 * i + 1] += I * Sg * gi * mine.lnTr;
                }
            }
            line_gr += I * Sg * shfl64(mine.dga_dgr, c);
            line_n += I * Sg * ga * shfl64(mine.lnTr, c);
        }
        if (lane == 0) {
            if (d_gref_line) d_gref_line[l] = accumulate ? d_gref_line[l] + line_gr : line_gr;
            if (d_n_line) d_n_line[l] = accumulate ? d_n_line[l] + line_n : line_n;
        }
    }
    if (lane < nc) {
        s_part[warp][lane][0] = accT;
        s_part[warp][lane][1] = accP;
        s_part[warp][lane][2] = accS;
        s_part[warp][lane][3] = accN;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nc * NQ; i += blockDim.x) {
        const int c = i / NQ, q = i % NQ;
        double s = 0.0;
        for (int w = 0; w < VW; ++w) s += q < 4 ? s_part[w][c][q] : s_broad[w][c][q - 4];
        block_part[((size_t)blockIdx.x * nc + c) * NQ + q] = s;
    }
}

// sum the block partials in a fixed order: quantity q of this chunk's condition c (values
// [blk][nc][NQ]) -> its output row (rows[c], or c0 + c when rows is null).  acc holds per
// row: gamma_scale and n_shift sums, then 2 nb per-broadener sums.
__global__ void __launch_bounds__(128) k_vjp_finish(const double *block_part, int n_blocks, int nc, int NQ, int c0,
                                                    const CParam *rows, double *dT, double *dP, double *acc) {
    // one warp per sum: lane j takes blocks j, j + 32, ..., then a fixed butterfly
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * 4 + (threadIdx.x >> 5);
    if (i >= nc * NQ) return;
    const int c = i / NQ, q = i % NQ;
    double s = 0.0;
    for (int b = lane; b < n_blocks; b += 32) s += block_part[((size_t)b * nc + c) * NQ + q];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane) return;
    const int r = rows ? rows[c].row : c0 + c;
    if (q == 0) dT[r] = s;
    else if (q == 1) dP[r] = s;
    else acc[(size_t)r * (NQ - 2) + (q - 2)] = s;
}

// global scalars and per-broadener sums: sums over conditions in order
__global__ void k_vjp_scalars(const double *acc, int nc, int nb, double *ds, double *dn, double *dg0b,
                              double *dnb) {
    const int q = threadIdx.x, W = 2 + 2 * nb;
    if (q >= W) return;
    double a = 0.0;
    for (int c = 0; c < nc; ++c) a += acc[(size_t)c * W + q];
    if (q == 0) {
        if (ds) *ds = a;
    } else if (q == 1) {
        if (dn) *dn = a;
    } else if (((q - 2) & 1) == 0) {
        if (dg0b) dg0b[(q - 2) / 2] = a;
    } else if (dnb) {
        dnb[(q - 2) / 2] = a;
    }
}

__global__ void k_to_f32(const double *in, float *out, size_t n) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        out[i] = (float)in[i];
}

// ---------------------------------------------------------------------------
// FP32 adjoint
// ---------------------------------------------------------------------------
// polynomial coefficient tables (ascending powers), derived at compile time from the
// published w4 coefficients of regions III and IV
template <int N>
struct Pc {
    double c[N];
};
template <int NA, int NB>
constexpr Pc<NA + NB - 1> pmul(const Pc<NA> &a, const Pc<NB> &b) {
    Pc<NA + NB - 1> r{};
    for (int i = 0; i < NA; ++i)
        for (int j = 0; j < NB; ++j) r.c[i + j] += a.c[i] * b.c[j];
    return r;
}
// a_i (k0 + k1 i): k0 = 1, k1 = 1 gives p + x p'; k0 = 0, k1 = 1 gives x p'
template <int N>
constexpr Pc<N> pidx(const Pc<N> &a, double k0, double k1) {
    Pc<N> r{};
    for (int i = 0; i < N; ++i) r.c[i] = a.c[i] * (k0 + k1 * i);
    return r;
}
template <int N>
constexpr Pc<N> psub(const Pc<N> &a, const Pc<N> &b) {
    Pc<N> r{};
    for (int i = 0; i < N; ++i) r.c[i] = a.c[i] - b.c[i];
    return r;
}
// region III: F = N3(t)/D3(t), t = y - i x
__device__ constexpr Pc<5> kN3{{16.4955, 20.20933, 11.96482, 3.778987, 0.5642236}};
__device__ constexpr Pc<6> kD3{{16.4955, 38.82363, 39.27121, 21.69274, 6.699398, 1.0}};
// d(tF)/dt = [D3 (N3 + t N3') - N3 (t D3')] / D3^2 (the t^9 coefficient cancels exactly)
__device__ constexpr Pc<10> kG3 = psub(pmul(kD3, pidx(kN3, 1.0, 1.0)), pmul(kN3, pidx(kD3, 0.0, 1.0)));
// region IV: F = e^u - t N4(m)/D4(m), u = t^2, m = -u (plain Horner in m)
__device__ constexpr Pc<7> kN4{{36183.31, 3321.9905, 1540.787, 219.0313, 35.76683, 1.320522, 0.56419}};
__device__ constexpr Pc<8> kD4{{32066.6, 24322.84, 9022.228, 2186.181, 364.2191, 61.57037, 1.841439, 1.0}};
// d(u r)/du = S4(m)/D4^2 with S4 = D4 (N4 + m N4_m) - N4 (m D4_m) (m^13 cancels exactly), and
// d(t r)/dt = r + 2 u r_u = T4(m)/D4^2 with T4 = D4 (N4 + 2 m N4_m) - N4 (2 m D4_m)
__device__ constexpr Pc<14> kS4 = psub(pmul(kD4, pidx(kN4, 1.0, 1.0)), pmul(kN4, pidx(kD4, 0.0, 1.0)));
__device__ constexpr Pc<14> kT4 = psub(pmul(kD4, pidx(kN4, 1.0, 2.0)), pmul(kN4, pidx(kD4, 0.0, 2.0)));

template <int N>
__device__ __forceinline__ Cx<float> horner_f(const Pc<N> &p, Cx<float> t, int top = N - 1) {
    Cx<float> r = cx<float>((float)p.c[top], 0.f);
#pragma unroll
    for (int i = N - 2; i >= 0; --i)
        if (i < top) r = (float)p.c[i] + r * t;
    return r;
}
// derivative of the polynomial: sum i c_i t^(i-1)
template <int N>
__device__ __forceinline__ Cx<float> dhorner_f(const Pc<N> &p, Cx<float> t) {
    Cx<float> r = cx<float>((float)((N - 1) * p.c[N - 1]), 0.f);
#pragma unroll
    for (int i = N - 2; i >= 1; --i) r = (float)(i * p.c[i]) + r * t;
    return r;
}

// Re F, Re F' and Re(F + t F') of w4 in regions II-IV at x >= 0, y (t = y - i x), FP32
__device__ __noinline__ float3 w4_band_f32(float x, float y) {
    constexpr double a = 1.410474, b = 0.5641896;
    const Cx<float> t = cx<float>(y, -x);
    const Cx<float> u = t * t;
    Cx<float> F, Fp, G;
    if (x + y >= 5.5f) {
        // region II: F = t (a + b u)/(3/4 + 3u + u^2)
        const Cx<float> D = 0.75f + u * (3.f + u);
        const Cx<float> iD = cdiv(cx<float>(1.f, 0.f), D);
        const Cx<float> iD2 = iD * iD;
        F = (t * ((float)a + (float)b * u)) * iD;
        Fp = ((float)(0.75 * a) + u * ((float)(2.25 * b - 3 * a) + u * ((float)(3 * b - 3 * a) + (float)(-b) * u))) * iD2;
        G = (2.f * t) * (((float)(0.75 * a) + u * ((float)(1.5 * b) + (float)(3 * b - a) * u)) * iD2);
    } else if (y >= 0.195f * x - 0.176f) {
        const Cx<float> N = horner_f(kN3, t), D = horner_f(kD3, t);
        const Cx<float> iD = cdiv(cx<float>(1.f, 0.f), D);
        const Cx<float> iD2 = iD * iD;
        F = N * iD;
        Fp = (dhorner_f(kN3, t) * D - N * dhorner_f(kD3, t)) * iD2;
        G = horner_f(kG3, t, 8) * iD2;
    } else {
        const Cx<float> m = cx<float>(-u.re, -u.im);
        const Cx<float> N = horner_f(kN4, m), D = horner_f(kD4, m);
        const Cx<float> iD = cdiv(cx<float>(1.f, 0.f), D);
        const Cx<float> iD2 = iD * iD;
        float sn, cs;
        sincosf(u.im, &sn, &cs);
        const float eu = expf(u.re);
        const Cx<float> e = cx<float>(eu * cs, eu * sn);
        F = e - t * (N * iD);
        Fp = (2.f * t) * e - horner_f(kT4, m) * iD2;
        G = e * (1.f + 2.f * u) - (2.f * t) * (horner_f(kS4, m, 12) * iD2);
    }
    return make_float3(F.re, Fp.re, G.re);
}

// compensated pair (hi + lo) and its exact-error addition (TwoSum), for warp reductions
struct F2 {
    float hi, lo;
};
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    const float s = __fadd_rn(a.hi, b.hi);
    const float bp = __fsub_rn(s, a.hi);
    const float err = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bp)), __fsub_rn(b.hi, bp));
    return F2{s, __fadd_rn(__fadd_rn(a.lo, b.lo), err)};
}
__device__ __forceinline__ F2 f2_warp_sum(F2 v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        F2 w{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
        v = f2_add(v, w);
    }
    return v;
}

__device__ __forceinline__ F2 f2_scale(F2 a, float k) {
    const float h = __fmul_rn(a.hi, k);
    return F2{h, fmaf(a.lo, k, fmaf(a.hi, k, -h))};
}
__device__ __forceinline__ F2 f2_of(const KahanF &k) { return F2{k.s, -k.c}; }

// Sums of one line and condition over grid points or block nodes, without their constant
// (q1 and q2 hold terms that fall as the fourth power of the distance: interpolated from 16 nodes these are
// good to 2.3e-6 of the value at a block's far end, 1.2e-7 of the near end's; q0's to 1.4e-8)
// factors, and the profile's constants in grid units.
template <int PROF>
struct VjpLine {
    float a_h, g_h, g2, C, g4, asc, y, thr2, ia2;
    const float *gx, *gw;
    int ngh;
    __device__ __forceinline__ VjpLine(float a, float g, const float *sx, const float *sw, int n)
        : a_h(a), g_h(g), gx(sx), gw(sw), ngh(n) {
        g2 = g * g;
        if (PROF == XC_VOIGT_W4) {
            asc = kSqrtLn2f * rcp_approx(a);                 // x = asc |delta|
            y = asc * g;
            C = a * a * (float)(0.5 / 0.6931471805599453) + g2;
            g4 = 4.f * g2;
            const float thr = (15.f - y) * rcp_approx(asc);
            thr2 = y < 15.f ? thr * thr : -1.f;              // region I iff u >= thr2
        } else if (PROF == XC_DOPPLER) {
            ia2 = rcp_approx(a * a);
        }
    }
    // one point (or node) at offset dl with weight gk
    __device__ __forceinline__ void add(float dl, float gk, float &q0, float &q1, float &q2) const {
        const float u = dl * dl;
        if (PROF == XC_VOIGT_W4) {
            const float t = C - u;
            const float rD = rcp_approx(fmaf(t, t, g4 * u));
            const float w = (u + C) * rD;
            q0 = fmaf(gk, w, q0);
            q1 = fmaf(gk, rD * fmaf(-2.f * t, w, 1.f), q1);
            q2 = fmaf(gk, u * w * rD, q2);
        } else if (PROF == XC_VOIGT_GH_BINNED) {
            // bin average of the Gauss-Hermite Voigt (Eq. e:sigma:quad), grid units (bin width 1):
            // per node j, s+ = delta + 1/2 - a x_j/sqrt(ln2), s- = s+ - 1, Q+- = s+-^2 + g^2,
            //   V = pi^(-3/2) sum_j w_j atan2(g, g^2 + s+ s-),
            //   dV/dg = pi^(-3/2) sum_j w_j (s+ s- - g^2)/(Q+ Q-),
            //   dV/da = pi^(-3/2) sum_j w_j (x_j/sqrt(ln2)) g (s+ + s-)/(Q+ Q-)
            const float d = dl + 0.5f;
            float v = 0.f, da = 0.f, dg = 0.f;
            for (int m = 0; m < ngh; ++m) {
                const float sp = fmaf(-a_h, gx[m], d), sm = sp - 1.f;
                const float Q = fmaf(sp, sp, g2) * fmaf(sm, sm, g2);
                const float iQ = Q > 1e-37f ? rcp_approx(Q) : 0.f;   // a pole at gamma = 0 (see gh_binned_deriv64)
                v = fmaf(gw[m], atan2_ypos(g_h, fmaf(sp, sm, g2)), v);
                dg = fmaf(gw[m], fmaf(sp, sm, -g2) * iQ, dg);
                da = fmaf(gw[m] * gx[m], (sp + sm) * iQ, da);
            }
            q0 = fmaf(gk, v, q0);
            q1 = fmaf(gk, da, q1);
            q2 = fmaf(gk, dg, q2);
        } else if (PROF == XC_DOPPLER) {
            // V = sqrt(ln2/pi)/a 2^(-u/a^2): sums of g 2^(-u/a^2) and g u 2^(-u/a^2)
            const float e = ex2_approx(-u * ia2) * gk;
            q0 += e;
            q1 = fmaf(e, u, q1);
        } else {
            // Lorentz: V = (1/pi) g/(u + g^2), dV/dg = (1/pi)(u - g^2)/(u + g^2)^2
            const float r = rcp_approx(u + g2);
            const float gr = gk * r;
            q0 += gr;
            q2 = fmaf(gr, (u - g2) * r, q2);
        }
    }
};

struct Vjp32Params {
    LinesDev L;
    size_t n;
    const int4 *geo;                      // per line: n, ka, kb (fixed cut), fraction (bits)
    const CParam *cp;                     // this launch's conditions, rows = caller index
    const CondDev *conds;                 // all conditions, caller order
    int nc;                               // conditions in this launch (<= 32)
    double nu_A, step, inv_step, cutoff, width_mult;
    int64_t n_pts;
    const float *g32;                     // dL/dsigma, [caller row][n_pts]
    double *block_part;                   // [block][nc][4 + 2 nb]
    double *d_gref_line, *d_n_line;       // per line (sorted order), nullable
    int accumulate;                       // add to the per-line outputs (later condition chunks)
    const double *ghx, *ghw;              // Gauss-Hermite nodes and weights (binned GH), device
    int ngh;
    const float *gnode;                   // dL/dsigma projected on the block nodes (see k_vjp_nodes), or nullptr
    int node_off[TR_LEVELS], nodes_per_cond;   // [caller row][nodes_per_cond], level l from node_off[l]
};

// dL/dsigma projected on the nodes of the blocks of xc_tree.cu: with V(k) = sum_m L_m(k) V(m)
// on a block, sum_k g_k V(k) = sum_m V(m) g(m), g(m) = sum_k L_m(k) g_k.  One CTA per
// 512-point block and condition: its eight 64-point blocks from the points, then the 128- and
// 512-point ones from those (the transposes of the sweep's matrices), in FP64.
__global__ void __launch_bounds__(128) k_vjp_nodes(const double *__restrict__ g, int64_t n_pts,
                                                   const double *__restrict__ mat, float *gnode, int off0, int off1,
                                                   int off2, int per_cond) {
    __shared__ double sG[512], s0[128];
    const int j = blockIdx.x, t = threadIdx.x;
    const double *gc = g + (size_t)blockIdx.y * (size_t)n_pts;
    float *out = gnode + (size_t)blockIdx.y * per_cond;
    for (int i = t; i < 512; i += 128) sG[i] = 512 * (int64_t)j + i < n_pts ? gc[512 * (int64_t)j + i] : 0.0;
    __syncthreads();
    {
        const int b = t >> 4, m = t & 15;
        double s = 0.0;
        for (int k = 0; k < 64; ++k) s = fma(mat[TR_MAT_PT + m * 64 + k], sG[64 * b + k], s);
        s0[t] = s;
        out[off0 + j * 128 + t] = (float)s;
    }
    __syncthreads();
    if (t < 64) {
        const int b = t >> 4, m = t & 15;
        double s = 0.0;
        for (int i = 0; i < 32; ++i) s = fma(mat[TR_MAT_128 + ((i >> 4) * TR_M + m) * TR_M + (i & 15)], s0[32 * b + i], s);
        out[off1 + j * 64 + t] = (float)s;
    } else if (t < 80) {
        const int m = t - 64;
        double s = 0.0;
        for (int i = 0; i < 128; ++i) s = fma(mat[TR_MAT_512 + ((i >> 4) * TR_M + m) * TR_M + (i & 15)], s0[i], s);
        out[off2 + j * 16 + m] = (float)s;
    }
}

// MIX: the Lorentz widths come from the handle's mixture of broadeners (per broadener
// and line rho_i gamma_0,i and n_i): gamma = gamma_scale P/P_ref sum_i rho_i gamma_0,i
// (T_ref/T)^(n_i + n_shift), and the adjoint also sums, per broadener, the gradients of a
// scale on its gamma_0 values (d gamma = gamma_i) and of a shift of its n values
// (d gamma = gamma_i ln(T_ref/T))
// WL: width-limited cuts (their code costs the fixed cut's kernel registers that it does not have)
// FAR: far points by the block nodes.  Without it (sparse lists, see route_adjoint_blocks) the points of
// a line are all there is, eight of a lane's in flight at a time.
template <int PROF, bool MIX, bool WL, bool FAR>
__global__ void __launch_bounds__(VT, MIX || !FAR ? 2 : 3) k_vjp32(Vjp32Params p) {
    __shared__ double s_part[VW][VMAXC][4];
    __shared__ double s_broad[VW][VMAXC][MIX ? 2 * VMAXB : 1];
    __shared__ float s_gx[PROF == XC_VOIGT_GH_BINNED ? 64 : 1], s_gw[PROF == XC_VOIGT_GH_BINNED ? 64 : 1];
    __shared__ float s_node[TR_LEVELS][TR_M];
    // the outermost Gauss-Hermite node lies within sqrt(2 n + 2) (a_h / sqrt(ln 2)) of the centre
    const float s_ext = sqrtf(2.f * (float)p.ngh + 2.f) * 1.203f;
    if (threadIdx.x < TR_LEVELS * TR_M)
        s_node[threadIdx.x / TR_M][threadIdx.x % TR_M] = tr_node(tr_block(threadIdx.x / TR_M), threadIdx.x % TR_M);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (PROF == XC_VOIGT_GH_BINNED) {
        // the node shifts x_j / sqrt(ln2) (in units of the Doppler width) and the weights
        for (int j = threadIdx.x; j < p.ngh; j += blockDim.x) {
            s_gx[j] = (float)(p.ghx[j] / kSqrtLn2);
            s_gw[j] = (float)p.ghw[j];
        }
        __syncthreads();
    }
    const int nc = p.nc;
    const int nb = MIX ? p.L.n_broad : 0, NQ = 4 + 2 * nb;
    if (MIX)
        for (int q = 0; q < 2 * nb; ++q) s_broad[warp][lane][q] = 0.0;
    const float inv_h = (float)(1.0 / p.step);
    // this lane's condition: FP32 constants, and FP64 accumulators of its four scalars
    const bool mine = lane < nc;
    const CParam cc = p.cp[mine ? lane : 0];
    // width-limited cuts: FP64 constants of the conditions, formed once (formed for every line from the
    // condition, their logarithm, root and divisions were most of the kernel at short cuts: Lorentz, 1e6
    // points, 3e5 lines, 1 condition, 500 widths: 3.07 ms, 1.71 now)
    __shared__ int2 s_wk[WL ? VW : 1][VMAXC];    // cut ranges of the warp's line
    __shared__ double s_wl[WL ? VMAXC : 1][5];   // alpha / nu, ln(T_ref/T), gamma_scale, P/P_ref, n_shift
    float invT, dQQ, lnTr, fP, fS;
    {
        const CondDev cd = p.conds[cc.row];
        if (WL && warp == 0 && mine) {
            s_wl[lane][0] = alpha_coef(cd.T, cd.mass_da);
            s_wl[lane][1] = log(cd.T_ref / cd.T);
            s_wl[lane][2] = cd.gamma_scale;
            s_wl[lane][3] = cd.P / cd.P_ref;
            s_wl[lane][4] = cd.n_shift;
        }
        invT = (float)(1.0 / cd.T);
        dQQ = (float)(cd.dQdT / cd.Q);
        lnTr = (float)log(cd.T_ref / cd.T);
        fP = (float)(cd.gamma_scale / cd.P_ref);     // d(gamma_scale P/P_ref)/dP
        fS = (float)(cd.P / cd.P_ref);               // d(gamma_scale P/P_ref)/d(gamma_scale)
    }
    if (WL) __syncthreads();
    double accT = 0.0, accP = 0.0, accS = 0.0, accN = 0.0;
    for (size_t l = (size_t)blockIdx.x * VW + warp; l < p.n; l += (size_t)gridDim.x * VW) {
        const float nu = (float)p.L.nu[l];
        const float E = p.L.elower[l];
        const float gA = (float)p.L.g_up[l] * p.L.A[l];
        const float gref = p.L.gamma_ref[l], nT = p.L.n_T[l];
        // lane c: intensity (scaled as the forward kernels scale it), widths in grid steps,
        // d ln I / dT = c2 E''/T^2 - (c2 nu/T^2)/(exp(c2 nu/T) - 1) - Q'/Q
        // gq: gamma/h per unit of gamma_scale P/P_ref; ngh: sum of (n + n_shift) gamma/h over
        // the width's terms (-T/h dgamma/dT); gi: the mixture's terms (per unit of gamma_scale P/P_ref)
        float Is = 0.f, ah = 1.f, gh = 0.f, tn = 0.f, dlnI = 0.f, gq = 0.f, ngh = 0.f;
        float gi[MIX ? VMAXB : 1];
        if (mine) {
            const float z = fmaf(E, cc.kT_hi, E * cc.kT_lo);
            const float xs = cc.c2T * nu;
            Is = cc.pref * gA * rcp_approx(nu * nu) * exp2_neg(z) * (-expm1f(-xs));
            if (MIX) {
                ah = __fmul_rn(cc.acoef * nu, inv_h);
                float nq = 0.f;
#pragma unroll
                for (int i = 0; i < VMAXB; ++i) {
                    gi[i] = 0.f;
                    if (i < nb) {
                        const float ni = (float)p.L.bn[(size_t)i * p.L.bstride + l] + cc.nshift;
                        gi[i] = (float)p.L.bgam[(size_t)i * p.L.bstride + l] * ex2_approx(ni * cc.log2Tr) * inv_h;
                        gq += gi[i];
                        nq = fmaf(ni, gi[i], nq);
                    }
                }
                gh = cc.pscale * gq;
                ngh = cc.pscale * nq;
            } else {
                line_widths(nu, gref, nT, cc, inv_h, &ah, &gh);
                tn = ex2_approx((nT + cc.nshift) * cc.log2Tr);
                gq = gref * tn * inv_h;
                ngh = gh * (nT + cc.nshift);
            }
            dlnI = cc.c2T * E * invT - xs * invT / expm1f(xs) - dQQ;
        }
        const int4 geo = p.geo[l];
        const int na = geo.x;
        const float ff = __int_as_float(geo.w);
        int ka = geo.y, kb = geo.z;
        // lane c: the cut min(cutoff, width_mult max(alpha, gamma)) of its condition, FP64 as in the
        // forward kernels' geometry
        if (WL) __syncwarp();   // the last line's ranges are no longer read
        if (WL && mine) {
            const double nud = p.L.nu[l], al = s_wl[lane][0] * nud, ns = s_wl[lane][4], lr = s_wl[lane][1];
            const double ga = MIX ? mixture_gamma64(p.L, l, ns, lr, s_wl[lane][2] * s_wl[lane][3])
                                  : s_wl[lane][2] * f2d(gref) * exp64((f2d(nT) + ns) * lr) * s_wl[lane][3];
            int64_t k0, k1;
            line_k_range(nud, fmin(p.width_mult * fmax(al, ga), p.cutoff), p.nu_A, p.step, p.inv_step, p.n_pts, &k0, &k1);
            s_wk[warp][lane] = make_int2((int)k0, (int)k1);
        }
        if (WL) __syncwarp();
        float SIm = 0.f, Sam = 0.f, Sgm = 0.f;   // lane c: its condition's three sums
        for (int c = 0; c < nc; ++c) {
            const float a_h = __shfl_sync(0xffffffffu, ah, c), g_h = __shfl_sync(0xffffffffu, gh, c);
            if (WL) {
                ka = s_wk[warp][c].x;
                kb = s_wk[warp][c].y;
            }
            const float *gc = p.g32 + (size_t)__shfl_sync(0xffffffffu, cc.row, c) * (size_t)p.n_pts;
            KahanF K0, K1, K2, B0, B1, B2;
            const VjpLine<PROF> ln_c(a_h, g_h, s_gx, s_gw, p.ngh);
            int k0 = ka, k1 = kb;   // the points around the centre, taken one by one
            if (PROF == XC_DOPPLER) {
                // 2^(-u / a^2) is exactly 0 in FP32 beyond 11.3 a
                const int r = (int)fminf(ceilf(11.3f * a_h) + 2.f, 1e9f);
                k0 = max(k0, na - r);
                k1 = (int)i64min(k1, (int64_t)na + r);
            } else if (FAR) {
                // The far points on both sides by the nodes of the blocks they fill: a block of
                // level l when it lies inside the cut and beyond the level's radius (xc_tree.cu).
                // Lane 5 s + q (s: side) finds segment q of that side: level 0 outside and inside
                // of level 1, level 1 outside and inside of level 2, level 2.
                const float *gn = p.gnode + (size_t)__shfl_sync(0xffffffffu, cc.row, c) * (size_t)p.nodes_per_cond;
                const float am = fminf(a_h, 1e6f);
                const int e = PROF == XC_VOIGT_W4 ? 2 + (int)ceilf(0.86f * am)
                              : PROF == XC_VOIGT_GH_BINNED ? 3 + (int)ceilf(am * s_ext)
                                                           : 1;
                const int core = PROF == XC_VOIGT_W4 ? 2 + (int)ceilf(18.05f * am) : 0;
                int A[TR_LEVELS], Z[TR_LEVELS];
#pragma unroll
                for (int l = 0; l < TR_LEVELS; ++l) {
                    const int D = max(tr_gap(l) + e, core), sh = l == 2 ? 9 : 6 + l;
                    const int lo = lane >= 5 ? max(ka, na + D + 1) : ka, hi = lane >= 5 ? kb : min(kb, na - D - 1);
                    A[l] = (lo + (1 << sh) - 1) >> sh;
                    Z[l] = (hi + 1) >> sh;
                }
                const bool h0 = Z[0] > A[0], h1 = h0 && Z[1] > A[1], h2 = h1 && Z[2] > A[2];
                const int q = lane >= 5 ? lane - 5 : lane;
                int lev = q < 2 ? 0 : (q < 4 ? 1 : 2), j0 = 0, j1 = 0;
                if (q == 0 && h0) { j0 = A[0]; j1 = h1 ? 2 * A[1] : Z[0]; }
                if (q == 1 && h1) { j0 = 2 * Z[1]; j1 = Z[0]; }
                if (q == 2 && h1) { j0 = A[1]; j1 = h2 ? 4 * A[2] : Z[1]; }
                if (q == 3 && h2) { j0 = 4 * Z[2]; j1 = Z[1]; }
                if (q == 4 && h2) { j0 = A[2]; j1 = Z[2]; }
                float q0 = 0.f, q1 = 0.f, q2 = 0.f;
                for (unsigned segs = __ballot_sync(0xffffffffu, lane < 10 && j1 > j0); segs; segs &= segs - 1) {
                    const int src = __ffs(segs) - 1;
                    const int lv = __shfl_sync(0xffffffffu, lev, src), sh = lv == 2 ? 9 : 6 + lv;
                    const int i1 = TR_M * __shfl_sync(0xffffffffu, j1, src);
                    const float *gl = gn + p.node_off[lv];
                    for (int i = TR_M * __shfl_sync(0xffffffffu, j0, src) + lane; i < i1; i += 32)
                        ln_c.add(((float)(((i >> 4) << sh) - na) + s_node[lv][i & 15]) - ff, gl[i], q0, q1, q2);
                }
                K0.add(q0);
                K1.add(q1);
                K2.add(q2);
                // what is left between the cut's ends and the blocks
                const bool hl = __shfl_sync(0xffffffffu, (int)h0, 0), hr = __shfl_sync(0xffffffffu, (int)h0, 5);
                const int l0 = 64 * __shfl_sync(0xffffffffu, A[0], 0), l1 = 64 * __shfl_sync(0xffffffffu, Z[0], 0);
                const int r0 = 64 * __shfl_sync(0xffffffffu, A[0], 5), r1 = 64 * __shfl_sync(0xffffffffu, Z[0], 5);
                const int nl = hl ? l0 - ka : 0, nr = hr ? kb - r1 + 1 : 0;
                q0 = q1 = q2 = 0.f;
                for (int i = lane; i < nl + nr; i += 32) {
                    const int k = i < nl ? ka + i : r1 + i - nl;
                    ln_c.add((float)(k - na) - ff, gc[k], q0, q1, q2);
                }
                K0.add(q0);
                K1.add(q1);
                K2.add(q2);
                if (hl) k0 = l1;
                if (hr) k1 = r0 - 1;
            }
            constexpr int U = FAR || PROF == XC_DOPPLER ? 1 : (PROF == XC_VOIGT_GH_BINNED ? 2 : 8);
            for (int k8 = k0 + lane; k8 <= k1; k8 += 32 * 8) {
                float q0 = 0.f, q1 = 0.f, q2 = 0.f;
#pragma unroll U
                for (int j = 0; j < 8; ++j) {
                    const int k = k8 + 32 * j;
                    if (k <= k1) {
                        const float d = (float)(k - na) - ff, gk = gc[k];
                        if (PROF != XC_VOIGT_W4 || d * d >= ln_c.thr2) {
                            ln_c.add(d, gk, q0, q1, q2);
                        } else {
                            const float3 r = w4_band_f32(ln_c.asc * fabsf(d), ln_c.y);
                            B0.add(gk * r.x);
                            B1.add(gk * r.z);   // Re(F + t F')
                            B2.add(gk * r.y);   // Re F'
                        }
                    } else if (U == 1) {
                        break;
                    }
                }
                K0.add(q0);
                K1.add(q1);
                K2.add(q2);
            }
            // the lanes' sums to the three derivative sums, each reduced over the warp
            F2 vI, va, vg;
            if (PROF == XC_VOIGT_W4) {
                const float ia = rcp_approx(a_h), g2 = g_h * g_h;
                const float kd = kSqrtLn2OverPi * ia;                        // sqrt(ln2/pi)/a
                const float kg = (float)(0.6931471805599453 / 1.772453850905516027) * ia * ia;
                vI = f2_add(f2_scale(f2_of(K0), kKappa * g_h), f2_scale(f2_of(B0), kd));
                va = f2_add(f2_scale(f2_of(K1), kKappa * g_h * (a_h * (float)(1.0 / 0.6931471805599453))),
                            f2_scale(f2_of(B1), -kd * ia));
                const F2 t = f2_add(f2_of(K1), f2_scale(f2_of(K2), -4.f));
                vg = f2_add(f2_add(f2_scale(f2_of(K0), kKappa), f2_scale(t, 2.f * kKappa * g2)), f2_scale(f2_of(B2), kg));
            } else {
                vI = f2_of(K0);
                va = f2_of(K1);
                vg = f2_of(K2);
            }
            vI = f2_warp_sum(vI);
            if (PROF != XC_LORENTZ) va = f2_warp_sum(va);
            if (PROF != XC_DOPPLER) vg = f2_warp_sum(vg);
            if (lane == c) {
                const float S0 = vI.hi + vI.lo, S1 = va.hi + va.lo, S2 = vg.hi + vg.lo;
                if (PROF == XC_VOIGT_W4) {
                    SIm = S0;
                    Sam = S1;
                    Sgm = S2;
                } else if (PROF == XC_VOIGT_GH_BINNED) {
                    constexpr float kpi = (float)(1.0 / (3.141592653589793 * 1.772453850905516));   // pi^(-3/2)
                    SIm = kpi * S0;
                    Sam = kpi * g_h * S1;
                    Sgm = kpi * S2;
                } else if (PROF == XC_DOPPLER) {
                    const float ia = rcp_approx(a_h);
                    const float pd = kSqrtLn2OverPi * ia;
                    SIm = pd * S0;
                    Sam = pd * (-S0 * ia + (float)(2.0 * 0.6931471805599453) * rcp_approx(a_h * a_h) * ia * S1);
                    Sgm = 0.f;
                } else {
                    SIm = g_h * (float)(1.0 / kPi) * S0;
                    Sam = 0.f;
                    Sgm = (float)(1.0 / kPi) * S2;
                }
            }
        }
        // lane c: this line's contributions to its condition (grid-unit sums: sum g V = SI/h,
        // sum g dV/dalpha = Sa/h^2, sum g dV/dgamma = Sg/h^2; alpha = a h, gamma = g h)
        double lg = 0.0, ln = 0.0;
        if (mine) {
            const float IS = Is * Sgm;
            accT += (double)(Is * (SIm * dlnI + Sam * ah * (0.5f * invT) - Sgm * ngh * invT));
            accP += (double)(IS * fP * gq);
            accS += (double)(IS * fS * gq);
            accN += (double)(IS * gh * lnTr);
            if (MIX) {
#pragma unroll
                for (int i = 0; i < VMAXB; ++i)
                    if (i < nb) {
                        const float t = IS * cc.pscale * gi[i];
                        s_broad[warp][lane][2 * i] += (double)t;
                        s_broad[warp][lane][2 * i + 1] += (double)(t * lnTr);
                    }
            } else {
                lg = (double)(IS * cc.pscale * tn) * cc.inv_scale;            // x 1/h^2 below
                ln = (double)(IS * gh * lnTr) * cc.inv_scale;                 // x 1/h below
            }
        }
        if (!MIX && (p.d_gref_line || p.d_n_line)) {
            for (int o = 1; o < nc; o <<= 1) {
                lg += __shfl_xor_sync(0xffffffffu, lg, o);
                ln += __shfl_xor_sync(0xffffffffu, ln, o);
            }
            if (lane == 0) {
                const double ih = 1.0 / p.step;
                lg *= ih * ih;
                ln *= ih;
                if (p.d_gref_line) p.d_gref_line[l] = p.accumulate ? p.d_gref_line[l] + lg : lg;
                if (p.d_n_line) p.d_n_line[l] = p.accumulate ? p.d_n_line[l] + ln : ln;
            }
        }
    }
    const double sc = cc.inv_scale / p.step;   // the intensity scale and the common 1/h
    if (mine) {
        s_part[warp][lane][0] = accT * sc;
        s_part[warp][lane][1] = accP * sc;
        s_part[warp][lane][2] = accS * sc;
        s_part[warp][lane][3] = accN * sc;
        if (MIX)
            for (int q = 0; q < 2 * nb; ++q) s_broad[warp][lane][q] *= sc;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nc * NQ; i += blockDim.x) {
        const int c = i / NQ, q = i % NQ;
        double sum = 0.0;
        for (int w = 0; w < VW; ++w) sum += q < 4 ? s_part[w][c][q] : s_broad[w][c][MIX ? q - 4 : 0];
        p.block_part[((size_t)blockIdx.x * nc + c) * NQ + q] = sum;
    }
}

typedef void (*VjpFn)(LinesDev, size_t, const CondDev *, int, double, double, int64_t, double, double,
                      const double *, double *, double *, double *, int, const double *, const double *, int);

static VjpFn pick(int prof) {
    switch (prof) {
    case XC_DOPPLER: return k_vjp_lines<XC_DOPPLER>;
    case XC_LORENTZ: return k_vjp_lines<XC_LORENTZ>;
    case XC_VOIGT_GH_BINNED: return k_vjp_lines<XC_VOIGT_GH_BINNED>;
    default: return k_vjp_lines<XC_VOIGT_W4>;
    }
}

#define VJ_TRY(call)                                                                            \
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

template <int PROF, bool FAR>
static void launch_vjp32(bool mix, bool wl, int blocks, cudaStream_t s, const Vjp32Params &p) {
    if (mix && wl) k_vjp32<PROF, true, true, FAR><<<blocks, VT, 0, s>>>(p);
    else if (mix) k_vjp32<PROF, true, false, FAR><<<blocks, VT, 0, s>>>(p);
    else if (wl) k_vjp32<PROF, false, true, FAR><<<blocks, VT, 0, s>>>(p);
    else k_vjp32<PROF, false, false, FAR><<<blocks, VT, 0, s>>>(p);
}
template <int PROF>
static void launch_vjp32(bool mix, bool wl, int blocks, cudaStream_t s, const Vjp32Params &p) {
    if (p.gnode) launch_vjp32<PROF, PROF != XC_DOPPLER>(mix, wl, blocks, s, p);
    else launch_vjp32<PROF, false>(mix, wl, blocks, s, p);
}

xc_status vjp_run(BatchedState *st, const VjpArgs &a, int64_t *launches) {
    cudaStream_t s = a.stream;
    const int nc = a.n_cond;
    const size_t n = a.n_lines, N = (size_t)a.grid.n;
    const bool f64 = a.opts.precision == XC_FP64_PLAIN;
    const bool host = a.mem == XC_MEM_HOST;
    int dev = 0, nsm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int blocks = (int)std::max<size_t>(1, std::min<size_t>((n + VW - 1) / VW, (size_t)nsm * 8));
    // scratch: [grad sigma in device memory][f32 copy][block partials][per-cond acc][outputs]
    //          FP32 path also: [per-line geometry n, f, ka, kb][line statistics][condition constants]
    size_t off = 0;
    auto carve = [&](size_t bytes) { size_t o = off; off += (bytes + 255) & ~size_t(255); return o; };
    size_t o_g = host ? carve((size_t)nc * N * 8) : 0;
    size_t o_g32 = f64 ? 0 : carve((size_t)nc * N * 4);
    const int nb = a.L.n_broad, NQ = 4 + 2 * nb;
    size_t o_bp = carve((size_t)blocks * VMAXC * NQ * 8);
    size_t o_acc = carve((size_t)nc * (NQ - 2) * 8);
    size_t o_out = host ? carve((size_t)(2 * nc + 2 + 2 * nb) * 8 + 2 * n * 8) : 0;
    size_t o_geo = f64 ? 0 : carve(n * 16);
    size_t o_gs = f64 ? 0 : carve(sizeof(GeomStats));
    size_t o_cp = f64 ? 0 : carve((size_t)nc * sizeof(CParam));
    // block nodes of the far field (FP32, lists that are dense enough): 208 floats per 512 points
    const bool far = !f64 && n && N &&
                     route_adjoint_blocks(a.opts.profile, a.opts.n_gh, a.opts.cutoff,
                                          route_cut_steps(a.opts.cutoff, a.opts.width_mult, a.grid, a.conds_host, nc),
                                          a.grid, a.reach, nc);
    const int nblk512 = far ? (int)((a.grid.n + 511) / 512) : 0;
    const size_t per_cond = (size_t)nblk512 * (128 + 64 + 16);
    size_t o_gn = far ? carve((size_t)nc * per_cond * 4) : 0;
    VJ_TRY(st->vjp_buf.ensure(off + 256));
    char *base = st->vjp_buf.as<char>();
    const double *g64 = a.grad_sigma;
    if (host && nc && N) {
        warm_host_pages(a.grad_sigma, (size_t)nc * N * 8);
        VJ_TRY(cudaMemcpyAsync(base + o_g, a.grad_sigma, (size_t)nc * N * 8, cudaMemcpyHostToDevice, s));
        g64 = (const double *)(base + o_g);
    }
    float *g32 = f64 ? nullptr : (float *)(base + o_g32);
    double *bp = (double *)(base + o_bp);
    double *acc = (double *)(base + o_acc);   // per condition row: scale, n-shift, per-broadener sums
    double *dT = a.dT, *dP = a.dP, *ds = a.d_gamma_scale, *dn = a.d_n_shift;
    double *dgl = a.d_gamma_ref_line, *dnl = a.d_n_line;
    double *dg0b = a.d_gamma0_broad, *dnb = a.d_n_broad;
    if (host) {
        double *o = (double *)(base + o_out);
        dT = o;
        dP = o + nc;
        ds = a.d_gamma_scale ? o + 2 * nc : nullptr;
        dn = a.d_n_shift ? o + 2 * nc + 1 : nullptr;
        dg0b = a.d_gamma0_broad ? o + 2 * nc + 2 : nullptr;
        dnb = a.d_n_broad ? o + 2 * nc + 2 + nb : nullptr;
        dgl = a.d_gamma_ref_line ? o + 2 * nc + 2 + 2 * nb : nullptr;
        dnl = a.d_n_line ? o + 2 * nc + 2 + 2 * nb + n : nullptr;
    }
    if (a.timing) cudaEventRecord(a.ev_begin, s);
    if (nc == 0 || n == 0) {
        if (nc) {
            VJ_TRY(cudaMemsetAsync(dT, 0, nc * 8, s));
            VJ_TRY(cudaMemsetAsync(dP, 0, nc * 8, s));
        }
        if (ds) VJ_TRY(cudaMemsetAsync(ds, 0, 8, s));
        if (dn) VJ_TRY(cudaMemsetAsync(dn, 0, 8, s));
        if (dg0b && nb) VJ_TRY(cudaMemsetAsync(dg0b, 0, nb * 8, s));
        if (dnb && nb) VJ_TRY(cudaMemsetAsync(dnb, 0, nb * 8, s));
        if (dgl && n) VJ_TRY(cudaMemsetAsync(dgl, 0, n * 8, s));
        if (dnl && n) VJ_TRY(cudaMemsetAsync(dnl, 0, n * 8, s));
    } else if (f64) {
        for (int c0 = 0; c0 < nc; c0 += VMAXC) {
            int cc = std::min(VMAXC, nc - c0);
            VjpFn fn = pick(a.opts.profile);
            fn<<<blocks, VT, 0, s>>>(a.L, n, a.conds_dev + c0, cc, a.grid.nu_A, a.grid.step, a.grid.n, a.opts.cutoff,
                                     a.opts.width_mult, g64 + (size_t)c0 * N, bp, dgl, dnl, c0 > 0 ? 1 : 0, a.ghx,
                                     a.ghw, a.opts.n_gh);
            k_vjp_finish<<<(cc * NQ + 3) / 4, 128, 0, s>>>(bp, blocks, cc, NQ, c0, nullptr, dT, dP, acc);
            *launches += 2;
        }
        k_vjp_scalars<<<1, 32, 0, s>>>(acc, nc, nb, ds, dn, dg0b, dnb);
        ++*launches;
        VJ_TRY(cudaGetLastError());
    } else {
        // FP32: the forward FP32 kernels' line geometry and condition constants, then the
        // adjoint per chunk of <= 32 conditions
        int4 *geo = (int4 *)(base + o_geo);
        GeomStats *gs = (GeomStats *)(base + o_gs);
        CParam *cp = (CParam *)(base + o_cp);
        if (N) {
            k_to_f32<<<nsm * 4, 256, 0, s>>>(g64, g32, (size_t)nc * N);
            ++*launches;
        }
        if (far) {
            const double *mat = nullptr;
            VJ_TRY(tree_mat(st, &mat, s));
            constexpr int kSlice = 65535;   // conditions of a launch: the grid's y limit
            for (int c0 = 0; c0 < nc; c0 += kSlice) {
                k_vjp_nodes<<<dim3(nblk512, std::min(kSlice, nc - c0)), 128, 0, s>>>(
                    g64 + (size_t)c0 * N, a.grid.n, mat, (float *)(base + o_gn) + (size_t)c0 * per_cond, 0, nblk512 * 128,
                    nblk512 * 192, (int)per_cond);
                ++*launches;
            }
        }
        VJ_TRY(launch_fp32_setup(a.L, n, a.conds_dev, nc, a.grid, a.opts.cutoff, geo, gs, cp, s));
        *launches += 2;
        for (int c0 = 0; c0 < nc; c0 += VMAXC) {
            Vjp32Params vp;
            vp.L = a.L;
            vp.n = n;
            vp.geo = geo;
            vp.cp = cp + c0;
            vp.conds = a.conds_dev;
            vp.nc = std::min(VMAXC, nc - c0);
            vp.nu_A = a.grid.nu_A;
            vp.step = a.grid.step;
            vp.inv_step = 1.0 / a.grid.step;
            vp.cutoff = a.opts.cutoff;
            vp.width_mult = a.opts.width_mult;
            vp.n_pts = a.grid.n;
            vp.g32 = g32;
            vp.block_part = bp;
            vp.d_gref_line = dgl;
            vp.d_n_line = dnl;
            vp.accumulate = c0 > 0 ? 1 : 0;
            vp.ghx = a.ghx;
            vp.ghw = a.ghw;
            vp.ngh = a.opts.n_gh;
            vp.gnode = far ? (const float *)(base + o_gn) : nullptr;
            vp.node_off[0] = 0;
            vp.node_off[1] = nblk512 * 128;
            vp.node_off[2] = nblk512 * 192;
            vp.nodes_per_cond = (int)per_cond;
            const bool mix = nb > 0;
            const bool wl = a.opts.width_mult > 0.0;
            switch (a.opts.profile) {
            case XC_DOPPLER: launch_vjp32<XC_DOPPLER>(mix, wl, blocks, s, vp); break;
            case XC_LORENTZ: launch_vjp32<XC_LORENTZ>(mix, wl, blocks, s, vp); break;
            case XC_VOIGT_GH_BINNED: launch_vjp32<XC_VOIGT_GH_BINNED>(mix, wl, blocks, s, vp); break;
            default: launch_vjp32<XC_VOIGT_W4>(mix, wl, blocks, s, vp); break;
            }
            k_vjp_finish<<<(vp.nc * NQ + 3) / 4, 128, 0, s>>>(bp, blocks, vp.nc, NQ, 0, cp + c0, dT, dP, acc);
            *launches += 2;
        }
        k_vjp_scalars<<<1, 32, 0, s>>>(acc, nc, nb, ds, dn, dg0b, dnb);
        ++*launches;
        VJ_TRY(cudaGetLastError());
    }
    if (a.timing) cudaEventRecord(a.ev_end, s);
    if (host) {
        if (nc) {
            VJ_TRY(cudaMemcpyAsync(a.dT, dT, nc * 8, cudaMemcpyDeviceToHost, s));
            VJ_TRY(cudaMemcpyAsync(a.dP, dP, nc * 8, cudaMemcpyDeviceToHost, s));
        }
        if (a.d_gamma_scale) VJ_TRY(cudaMemcpyAsync(a.d_gamma_scale, ds, 8, cudaMemcpyDeviceToHost, s));
        if (a.d_n_shift) VJ_TRY(cudaMemcpyAsync(a.d_n_shift, dn, 8, cudaMemcpyDeviceToHost, s));
        if (a.d_gamma0_broad && nb) VJ_TRY(cudaMemcpyAsync(a.d_gamma0_broad, dg0b, nb * 8, cudaMemcpyDeviceToHost, s));
        if (a.d_n_broad && nb) VJ_TRY(cudaMemcpyAsync(a.d_n_broad, dnb, nb * 8, cudaMemcpyDeviceToHost, s));
        if (a.d_gamma_ref_line && n) VJ_TRY(cudaMemcpyAsync(a.d_gamma_ref_line, dgl, n * 8, cudaMemcpyDeviceToHost, s));
        if (a.d_n_line && n) VJ_TRY(cudaMemcpyAsync(a.d_n_line, dnl, n * 8, cudaMemcpyDeviceToHost, s));
        VJ_TRY(cudaStreamSynchronize(s));
    }
    return XC_OK;
}

}  // namespace xc
