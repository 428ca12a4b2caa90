// xc_f32.cuh -- device code shared by the FP32 profile kernels: packed f32x2 arithmetic,
// the per-(line, condition) constants of every profile and the profile values.
#pragma once

#include <math.h>

#include "xc_batched.cuh"

namespace xc {

constexpr float kPiM32 = 0.17958712212516656f;          // pi^(-3/2)
constexpr float kFarU3 = 1.f / 0.003f;                   // 3-term far-wing series from u >= C / 0.003
constexpr float kFarU4 = 1.f / 0.012f;                   // 4-term far-wing series from u >= C / 0.012

// Two FP32 values in one 64-bit register pair, for the packed f32x2 arithmetic of
// sm_100-class GPUs: one instruction issue performs two FP32 adds / multiplies /
// FMAs (the FMA pipe throughput is unchanged; the issue slots are halved).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pk2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void upk2(f32x2 v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ float lo2(f32x2 v) { float a, b; upk2(v, a, b); return a; }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 rcp2(f32x2 a) {
    float x, y;
    upk2(a, x, y);
    return pk2(rcp_approx(x), rcp_approx(y));
}
// ---------------------------------------------------------------------------
// per-(line, condition) constants, by profile
//   W4 : A = {E', F', P', P'C'}   B = {a, y, Pv, thr^2}   (grid units)
//   VV : A = reference wing {E', F', P', P'C'} (or {a, -1, P, y} where it is not region I
//        throughout)   B = {a, y, Pv, exact-zone half-width}
//   LOR: A = {G', P', 0, 0}
//   DOP: A = {qd, Pd, 0, 0}
//   GHS: A = {sh, G', P, 0}
//   GHB: A = {sh, g', G' - 1/4, P}
// ---------------------------------------------------------------------------
// Voigt w4 zones of a (line, condition) from its widths in grid steps: x = a |delta|,
// y, the region-I threshold u >= t2 (t2 < 0: region I everywhere) and the far radius D.
// Explicitly rounded operations: every kernel that splits work by these gets the same bits.
//   Far wing: the region-I rational P (u + C)/(u^2 + E u + F) equals its series
//   P r (1 + c1 r + c2 r^2 + ...) in r = 1/u, c1 = C - E = 3b - g^2, c2 = E^2 - C E - F =
//   (g^2 - 5b)^2 - 20 b^2.  u^2 + E u + F has its two roots on |u| = C, so |c_n| <=
//   (2n + 1) C^n and the terms dropped beyond r^2 stay below 7 x^3 / (1 - 9x/7), x = C r:
//   at u >= C / 0.003 that is < 2e-7 of the value, below FP32 rounding of the rational;
//   with four terms (c3 = -E c2 - F c1) the bound is 9 x^4 / (1 - 11x/9) < 2e-7 from
//   u >= C / 0.012.
//   D3, D4: integer radii (grid steps) beyond which every point is in the 3- or 4-term
//   far zone and in region I; a block [t0, t1] with n - D > t1 or n + D < t0 (n =
//   integer part of the line position) qualifies.
struct W4Zone {
    float a, y, t2, D3, D4;
};
__device__ __forceinline__ W4Zone w4_zone(float ah, float gh) {
    W4Zone z;
    const float rah = rcp_approx(ah);
    z.a = __fmul_rn(kSqrtLn2f, rah);
    z.y = __fmul_rn(z.a, gh);
    const float thr = __fmul_rn(__fmul_rn(__fsub_rn(15.f, z.y), ah), 1.f / kSqrtLn2f);
    z.t2 = z.y < 15.f ? __fmul_rn(thr, thr) : -1.f;
    const float Crn = __fadd_rn(__fmul_rn(__fmul_rn(ah, ah), (float)(0.5 / 0.6931471805599453)), __fmul_rn(gh, gh));
    // any D >= sqrt(uf) is valid: approximate square root (one MUFU op), scaled up by
    // more than its error bound
    float sq3, sq4;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(sq3) : "f"(fmaxf(__fmul_rn(Crn, kFarU3), z.t2)));
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(sq4) : "f"(fmaxf(__fmul_rn(Crn, kFarU4), z.t2)));
    z.D3 = ceilf(__fmul_rn(sq3, 1.000001f)) + 1.f;
    z.D4 = ceilf(__fmul_rn(sq4, 1.000001f)) + 1.f;
    return z;
}

// S = (p0, p1, p2, D) of the 3-term far-wing series; D = D4 (the tensor-core kernel's
// radius) when that kernel takes the far wings (d4), else D3
static __device__ __noinline__ float w4_value_f32(float delta, const float4 &B);

// EXT: the options that change a line's constants per (line, condition) -- emission,
// intensity thresholds, broadener mixtures, VVN -- are honoured; without them (EXT = false)
// the Voigt-w4 hot kernels carry none of their checks
template <int PROF, bool EXT = true>
__device__ __forceinline__ void line_consts(const LinesDev &L, size_t l, const CParam &c, float h, float inv_h,
                                            float4 *A, float4 *B, float *thr2, float4 *S, bool d4 = false) {
    const float nu = (float)L.nu[l];
    const float E = L.elower[l];
    // Boltzmann factor exp(-c2 E/T) = 2^-(E c2 log2e / T), product kept to ~1 ulp
    float z = fmaf(E, c.kT_hi, E * c.kT_lo);
    float boltz = exp2_neg(z);
    float I;
    if (EXT && c.emis != 0.f) {
        // Eq. (e:emiss) times h c nu: the upper state's Boltzmann factor as exp(-c2 E''/T)
        // exp(-c2 nu/T), each to ~1 ulp
        I = c.pref * ((float)L.g_up[l] * L.A[l]) * nu * boltz * exp2_neg(fmaf(nu, c.kT_hi, nu * c.kT_lo));
    } else {
        float stim = -expm1f(-c.c2T * nu);
        I = c.pref * ((float)L.g_up[l] * L.A[l]) * rcp_approx(nu * nu) * boltz * stim;
    }
    // left out by the intensity threshold for this condition (decided in FP64)
    if (EXT && L.keep && !((L.keep[l * (size_t)L.keep_words + (c.row >> 5)] >> (c.row & 31)) & 1u)) I = 0.f;
    // VVN: this (line, condition)'s area normalisation (computed in FP64)
    if (EXT && L.vv_scale) I *= L.vv_scale[l * (size_t)L.vv_stride + c.row];
    float al = c.acoef * nu;                                                   // Eq. e:alphaD
    float ah, gh;                                                              // widths in grid steps
    if (EXT && L.gamma_lc) {
        // broadener mixture: the width of this (line, condition), computed in FP64
        ah = __fmul_rn(c.acoef * nu, inv_h);
        gh = __fmul_rn(L.gamma_lc[l * (size_t)L.gamma_stride + c.row], inv_h);
    } else {
        line_widths(nu, L.gamma_ref[l], L.n_T[l], c, inv_h, &ah, &gh);
    }
    *thr2 = -1.f;
    *S = make_float4(0.f, 0.f, 0.f, __int_as_float(0x7f800000));
    if (PROF == XC_VOIGT_W4) {
        float b = ah * ah * (float)(0.5 / 0.6931471805599453);
        float g2 = gh * gh;
        float C = b + g2;
        float P = I * kKappa * gh * inv_h;
        *A = make_float4(2.f * (g2 - b), C * C, P, P * C);
        // a, y and the region-I threshold decide which kernel evaluates a point (the
        // main kernel: |x| + y >= 15; the centre-zone kernel: the rest); the far radius
        // which points the tensor-core kernel takes (see w4_zone)
        const W4Zone z = w4_zone(ah, gh);
        float Pv = I * kSqrtLn2OverPi * rcp_approx(al);
        *B = make_float4(z.a, z.y, Pv, z.t2);
        *thr2 = z.t2;
        float e5 = g2 - 5.f * b;
        *S = make_float4(P, P * (3.f * b - g2), P * fmaf(e5, e5, -20.f * b * b), d4 ? z.D4 : z.D3);
    } else if (PROF == XC_LORENTZ) {
        *A = make_float4(fmaxf(gh * gh, 1e-30f), I * gh * inv_h * (float)(1.0 / 3.141592653589793), 0.f, 0.f);
    } else if (PROF == XC_DOPPLER) {
        float qd = rcp_approx(ah * ah);
        *A = make_float4(qd, I * kSqrtLn2OverPi * rcp_approx(al), 0.f, 0.f);
    } else if (PROF == XC_VOIGT_GH_SAMPLED) {
        *A = make_float4(ah / kSqrtLn2f, fmaxf(gh * gh, 1e-30f), I * kPiM32 * gh * inv_h, 0.f);
    } else if (PROF == XC_VOIGT_VV) {
        // B: the line's own w4 Voigt (a, y, Pv) and the exact zone's half-width in grid steps;
        // A: the reference wing -- the Voigt of a line at 1 cm^-1, Doppler HWHM alpha / nu:
        // a_ref = a nu, y_ref = a_ref g, amplitude Pv nu, times beta (Eq. e:beta) when asked
        const float a = kSqrtLn2f * rcp_approx(ah), y = a * gh;
        const float Pv = I * kSqrtLn2OverPi * rcp_approx(al);
        const float ar = a * nu, yr = ar * gh;
        const float sp = c.vv_split * inv_h;
        float Pw = Pv * nu;
        if (c.vv_beta) {
            const float rw = w4_value_f32(sp, make_float4(ar, yr, 1.f, 0.f));
            Pw = rw > 0.f ? w4_value_f32(sp, make_float4(a, y, Pv, 0.f)) / rw : 0.f;
        }
        if (ar * (sp + gh) >= 15.f) {
            // beyond the exact zone the reference Voigt is in w4's region I everywhere
            // (x_ref + y_ref > a_ref (sp + g) >= 15): its rational in u = delta^2, as the
            // Voigt w4 constants A (with b_ref = 1 / (2 a_ref^2), C = b_ref + g^2).
            // a_ref = sqrt(ln 2) h / (alpha / nu) does not depend on nu (thousands for common
            // steps), so only a split and a Lorentz width both far below a grid step fail it
            const float br = 0.5f * rcp_approx(ar * ar), g2 = gh * gh, Cr = br + g2;
            const float Pr = Pw * 0.5641896f * gh * rcp_approx(ar);
            *A = make_float4(2.f * (g2 - br), Cr * Cr, Pr, Pr * Cr);
        } else {
            *A = make_float4(ar, -1.f, Pw, yr);   // flagged by A.y < 0: the complex w4 where needed
        }
        *B = make_float4(a, y, Pv, sp);
    } else if (PROF == XC_DOPPLER_BINNED) {
        // Eq. (eqn:sig_ij) in grid steps: x+- = (sqrt(ln2)/ah) (delta +- 1/2), I/(2h)
        *A = make_float4(kSqrtLn2f * rcp_approx(ah), 0.5f * I * inv_h, 0.f, 0.f);
    } else if (PROF == XC_LORENTZ_BINNED) {
        // Eq. (eqn:sig_lor-2) in grid steps: y+- = (delta +- 1/2)/gh, I/(pi h)
        *A = make_float4(gh, gh * gh - 0.25f, I * inv_h * (float)(1.0 / 3.141592653589793), 0.f);
    } else {
        *A = make_float4(ah / kSqrtLn2f, gh, gh * gh - 0.25f, I * kPiM32 * inv_h);
    }
}

// Re w in w4's region II (5.5 <= |x| + y < 15) in real arithmetic.  The region-II
// rational t(a + b t^2)/(t^4 + 3 t^2 + 3/4) has denominator (t^2 + Q1)(t^2 + Q2) with
// Q1,2 = (3 -+ sqrt 6)/2, so it splits into two partial fractions A_m t/(t^2 + Q_m),
// A_m = (a - b Q_m)/(Q_other - Q_m); each is a pair of Lorentzians in x at +-sqrt(Q_m):
//   Re w = y sum_m A_m (X + Y + Q_m) / ((X + Y - Q_m)^2 + 4 Q_m Y),  X = x^2, Y = y^2.
// (The nodes +-sqrt(Q_m) are those of 4-point Gauss-Hermite quadrature.)
__device__ __forceinline__ float w4_region2_re(float x, float y) {
    constexpr double a = 1.410474, b = 0.5641896, s6 = 2.449489742783178098;
    constexpr float Q1 = (float)((3.0 - s6) / 2.0), Q2 = (float)((3.0 + s6) / 2.0);
    constexpr float A1 = (float)((a - b * ((3.0 - s6) / 2.0)) / s6);
    constexpr float A2 = (float)(-(a - b * ((3.0 + s6) / 2.0)) / s6);
    float X = x * x, Y = y * y;
    float t1 = X + Y - Q1, t2 = X + Y - Q2;
    float D1 = fmaf(t1, t1, 4.f * Q1 * Y), D2 = fmaf(t2, t2, 4.f * Q2 * Y);
    float N1 = A1 * (X + Y + Q1), N2 = A2 * (X + Y + Q2);
    return y * fmaf(N1, D2, N2 * D1) * rcp_approx(D1 * D2);
}

// full FP32 w4 Voigt value (all regions) times Pv, at grid offset delta
// (kept out of line: only the few points with |x| + y < 5.5 reach it, and inlining
// its four regions into every unrolled (point, condition) slot bloats the kernel)
static __device__ __noinline__ float w4_value_f32(float delta, const float4 &B) {
    float x = B.x * fabsf(delta);
    Cx<float> w = w4_eval<float>(x, B.y, nullptr);
    return B.z * w.re;
}

// Re w in w4's region I from (x, y): 0.5641896 y (0.5 + X + Y) / ((X + Y - 0.5)^2 + 2Y)
__device__ __forceinline__ float w4_region1_re(float x, float y) {
    float X = x * x, Y = y * y;
    float t = X + Y - 0.5f;
    return 0.5641896f * y * (0.5f + X + Y) * rcp_approx(fmaf(t, t, 2.f * Y));
}

// Binned Gauss-Hermite Voigt where t = g / (s+ s- + g^2) <= kGhFarT at every node: atan(t) =
// t - t^3/3 + t^5/5, the rest below t^6 / 7 = 1e-10 of it, instead of the general arctangent
// (20 instructions a node).  gh_far: whether a line qualifies beyond `gap` grid steps of its
// centre, its outermost node lying within ext of it.
constexpr float kGhFarT = 0.03f;
__device__ __forceinline__ bool gh_far(float g, float gap, float ext) {
    const float d = gap - ext - 1.f;
    return d > 0.f && g <= kGhFarT * d * d;
}
__device__ __forceinline__ float gh_far_value(float delta, const float4 &A, const float *s_x, const float *s_w, int ngh) {
    float s = 0.f;
#pragma unroll 4
    for (int j = 0; j < ngh; ++j) {
        const float e = fmaf(-A.x, s_x[j], delta);
        const float t = A.y * rcp_approx(fmaf(e, e, A.z));
        const float q = t * t;
        s = fmaf(s_w[j], t * fmaf(q, fmaf(q, 0.2f, -1.f / 3.f), 1.f), s);
    }
    return A.w * s;
}

template <int PROF>
__device__ __forceinline__ float contrib_single(float u, float delta, const float4 &A, const float4 &B,
                                                const float *s_x, const float *s_w, int ngh) {
    if (PROF == XC_VOIGT_W4) {
        // region I only; points with |x| + y < 15 belong to the centre-zone kernel
        float D = fmaf(u, u + A.x, A.y);
        float q = fmaf(A.z, u, A.w);
        return u >= B.w ? q * rcp_approx(D) : 0.f;
    } else if (PROF == XC_LORENTZ) {
        return A.y * rcp_approx(u + A.x);
    } else if (PROF == XC_DOPPLER) {
        return A.y * ex2_approx(-A.x * u);
    } else if (PROF == XC_VOIGT_GH_SAMPLED) {
        float s = 0.f;
        for (int j = 0; j < ngh; ++j) {
            float e = fmaf(-A.x, s_x[j], delta);
            s = fmaf(s_w[j], rcp_approx(fmaf(e, e, A.y)), s);
        }
        return A.z * s;
    } else if (PROF == XC_VOIGT_VV) {
        // Eq. (e:fast-v): the line's own Voigt in the exact zone, the reference wing beyond it.
        // Both are w4 Voigts.  The reference wing (most of the points) is region I throughout
        // for almost every line: its rational in u with the line's constants, as Voigt w4's
        // main kernel evaluates it; in the exact zone w4 is its region-I rational in real
        // form where |x| + y >= 15 and the full w4 only for the few points nearer the centre
        const float ad = fabsf(delta);
        if (ad > B.w) {
            if (A.y >= 0.f) return fmaf(A.z, u, A.w) * rcp_approx(fmaf(u, u + A.x, A.y));
            const float x = A.x * ad;
            return x + A.w >= 15.f ? A.z * w4_region1_re(x, A.w) : w4_value_f32(delta, make_float4(A.x, A.w, A.z, 0.f));
        }
        const float x = B.x * ad;
        return x + B.y >= 15.f ? B.z * w4_region1_re(x, B.y) : w4_value_f32(delta, make_float4(B.x, B.y, B.z, 0.f));
    } else if (PROF == XC_DOPPLER_BINNED) {
        // erf(x+) - erf(x-) on the side |delta| of the (symmetric) profile, as
        // erfc(x-) - erfc(x+): no difference of two numbers near 1 in the wings
        const float t = fabsf(delta);
        return A.y * (erfcf(A.x * (t - 0.5f)) - erfcf(A.x * (t + 0.5f)));
    } else if (PROF == XC_LORENTZ_BINNED) {
        // atan(y+) - atan(y-) = atan2(y+ - y-, 1 + y+ y-), both arguments scaled by gh^2 > 0
        return A.z * atan2_ypos(A.x, u + A.y);
    } else {
        float s = 0.f;
        for (int j = 0; j < ngh; ++j) {
            float e = fmaf(-A.x, s_x[j], delta);
            s = fmaf(s_w[j], atan2_ypos(A.y, fmaf(e, e, A.z)), s);
        }
        return A.w * s;
    }
}

// Re w in w4's region III (|x| + y < 5.5, y >= 0.195 |x| - 0.176): the real part of the quotient
__device__ __forceinline__ float w4_region3_re(float x, float y) {
    // N(t) and D(t) have real coefficients: synthetic division by (z - t)(z - conj t) =
    // z^2 - r z + s takes two operations per coefficient instead of the four of a complex
    // Horner step, and is no less accurate here (rms error against FP64 over region III
    // 2.2e-7, complex Horner 2.4e-7; in region IV it would be 6 times worse, so not there)
    const float r = y + y, s = fmaf(x, x, y * y);
    const float n3 = fmaf(0.5642236f, r, 3.778987f);
    const float n2 = fmaf(r, n3, fmaf(-s, 0.5642236f, 11.96482f));
    const float n1 = fmaf(r, n2, fmaf(-s, n3, 20.20933f));
    const float d4 = r + 6.699398f;
    const float d3 = fmaf(r, d4, 21.69274f - s);
    const float d2 = fmaf(r, d3, fmaf(-s, d4, 39.27121f));
    const float d1 = fmaf(r, d2, fmaf(-s, d3, 38.82363f));
    const float Nr = fmaf(y, n1, fmaf(-s, n2, 16.4955f)), Dr = fmaf(y, d1, fmaf(-s, d2, 16.4955f));
    const float Ni = x * n1, Di = x * d1;   // both imaginary parts with the sign of conj t
    return fmaf(Nr, Dr, Ni * Di) * recip(fmaf(Dr, Dr, Di * Di));
}

// Re w in w4's region IV (|x| + y < 5.5, y < 0.195 |x| - 0.176): cos(Im u) of exp(u), u = t^2,
// and no sine
__device__ __forceinline__ float w4_region4_re(float x, float y) {
    const Cx<float> t = cx<float>(y, -x);
    const Cx<float> u = t * t;
    const Cx<float> m = cx<float>(-u.re, -u.im);
    const Cx<float> N = 36183.31f + m * (3321.9905f + m * (1540.787f + m * (219.0313f +
                        m * (35.76683f + m * (1.320522f + 0.56419f * m)))));
    const Cx<float> D = 32066.6f + m * (24322.84f + m * (9022.228f + m * (2186.181f +
                        m * (364.2191f + m * (61.57037f + m * (1.841439f + m))))));
    const Cx<float> r = cdiv(N, D);
    return expf(u.re) * cosf(u.im) - (t.re * r.re - t.im * r.im);
}

__device__ __forceinline__ float w4_region34_re(float x, float y) {
    return y >= 0.195f * fabsf(x) - 0.176f ? w4_region3_re(x, y) : w4_region4_re(x, y);
}

// width of a condition's profiles at a representative line (nu = 5000 cm^-1, n = 0.6):
// C = alpha^2 / (2 ln 2) + gamma^2, the scale of the far-wing radius
__device__ inline double cond_width_key(const CondDev &d) {
    const double al = alpha_coef(d.T, d.mass_da) * 5000.0;
    const double ga = d.gamma_scale * (d.P / d.P_ref) * pow(d.T_ref / d.T, 0.6 + d.n_shift);
    return al * al * (0.5 / 0.6931471805599453) + ga * ga;
}

// Position of condition c in order of increasing profile width (stable), so that the
// conditions sharing a tile of the CUDA-core kernel have similar far-wing radii
__device__ inline int cond_rank(int c, const CondDev *conds, int n_cond) {
    const double key = cond_width_key(conds[c]);
    int rank = 0;
    for (int j = 0; j < n_cond; ++j) {
        const double kj = cond_width_key(conds[j]);
        rank += (kj < key) || (kj == key && j < c);
    }
    return rank;
}

// Per-condition constants in parts (their FP64 chains are independent of one another)
__device__ inline void cparam_strength(const CondDev &d, const GeomStats *gs, int quantity, CParam *p) {
    const bool emis = quantity == XC_EMISSION;
    const double pref = emis ? d.abundance * kPlanckErg * kLightCm / (4.0 * kPi * d.Q)
                             : d.abundance / (8.0 * kPi * kLightCm * d.Q);
    const double s1 = (double)__uint_as_float(gs->gA_nu2_bits);
    const double s2 = (double)__uint_as_float(gs->gA_nu_bits);
    const double numax = (double)__uint_as_float(gs->nu_bits);
    // bound on the largest intensity (absorption), or emissivity: g A nu <= max(g A / nu) nu_max^2
    const double ib = emis ? pref * s2 * numax * numax : pref * fmin(s1, kC2 / d.T * s2);
    int e2 = 0;
    if (ib > 0.0 && isfinite(ib)) e2 = max(-120, min(120, ilogb(1e10 / ib)));   // floor(log2)
    p->inv_scale = ldexp(1.0, -e2);
    p->pref = (float)(pref * ldexp(1.0, e2));
    p->emis = emis ? 1.f : 0.f;
}
__device__ inline void cparam_temperature(const CondDev &d, CParam *p) {
    const double kT = kC2 * 1.4426950408889634 / d.T;
    p->kT_hi = (float)kT;
    p->kT_lo = (float)(kT - (double)p->kT_hi);
    p->c2T = (float)(kC2 / d.T);
    p->nshift = (float)d.n_shift;
}
__device__ inline void cparam_widths(const CondDev &d, CParam *p) {
    p->acoef = (float)alpha_coef(d.T, d.mass_da);
    p->pscale = (float)(d.gamma_scale * d.P / d.P_ref);
}

// Per-condition constants of condition c; row keeps the caller's index.
__device__ inline CParam make_cparam(int c, const CondDev *conds, const GeomStats *gs, double step, int quantity,
                                     const unsigned *gmax_bits, float vv_split, int vv_beta) {
    const CondDev d = conds[c];
    CParam p;
    cparam_strength(d, gs, quantity, &p);
    cparam_temperature(d, &p);
    cparam_widths(d, &p);
    p.log2Tr = (float)log2(d.T_ref / d.T);
    p.row = c;
    p.vv_split = vv_split;
    p.vv_beta = vv_beta;
    {
        // D4 <= ceil(sqrt(max(C k4, t2))) + 1 grows with both widths; t2 <= (15 a_h / sqrt ln2)^2.
        // Upper bounds of the widths from the line statistics (|n| <= nT_max), with margin.
        const double num = (double)__uint_as_float(gs->nu_bits);
        const double grm = (double)__uint_as_float(gs->gref_bits);
        const double ntm = (double)__uint_as_float(gs->nT_bits);
        const double lr = log(d.T_ref / d.T);
        const double tf = fmax(exp((ntm + d.n_shift) * lr), exp((-ntm + d.n_shift) * lr));
        const double ah = alpha_coef(d.T, d.mass_da) * num / step;
        // under a broadener mixture the largest width of this condition over all lines
        const double gh = gmax_bits ? (double)__uint_as_float(gmax_bits[c]) / step
                                    : fabs(d.gamma_scale * d.P / d.P_ref) * grm * tf / step;
        const double C = ah * ah * (0.5 / 0.6931471805599453) + gh * gh;
        const double t2 = 225.0 * ah * ah / 0.6931471805599453;
        const double uf = fmax(C * (1.0 / 0.012), t2);
        const double db = ceil(sqrt(uf) * 1.001) + 3.0;
        p.dbound = (isfinite(db) && db < 1e9) ? (float)db : 1e9f;
    }
    return p;
}


// A timing event inside the sweep: while the sweep is captured into a graph it must be an
// external event node (a plain record would become an internal dependency); on a stream
// that is not capturing (the per-condition sweeps of a width-limited cut) the external
// flag is refused, and a plain record is the same thing.
static inline cudaError_t record_timing_event(cudaEvent_t ev, cudaStream_t s) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(s, &cs);
    if (e != cudaSuccess) return e;
    return cs == cudaStreamCaptureStatusActive ? cudaEventRecordWithFlags(ev, s, cudaEventRecordExternal)
                                               : cudaEventRecord(ev, s);
}

}  // namespace xc
