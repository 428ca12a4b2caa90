// xc_route.h -- which kernels run a call, from its sizes alone (host code without CUDA).
#pragma once

#include <math.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/xc.h"

namespace xc {

// FP64 blocks (xc_tree64.cu): every profile but the Vectorized Voigt, which is not smooth at its
// split.  Positions and candidate ranges are 32-bit integers: fewer than 2^30 points, a cut of
// fewer than 2^20 steps; beyond 2^30 lines the scratch would crowd out other buffers.
//   Fine steps: a point's wavenumber nu_A + k step is off its exact place by the rounding r of
// |nu|, which the blocks follow to first order: the rest is 3 (r / d)^2 of a value at distance d >=
// 60 steps, 2e-16 at r = 2^-21 steps.  Steps finer than that against |nu| go to the direct sum
// (nu_A + k step stops growing with k altogether where the step is below the rounding).
//   Long cuts: four lines to a reciprocal multiplies 16 powers of the distance, up to 1e15.
inline bool route_blocks64(int profile, const xc_grid &g, double cutoff, size_t n) {
    const double top = fmax(fabs(g.nu_A), fabs(g.nu_A + g.step * (double)g.n));
    return profile != XC_VOIGT_VV && cutoff / g.step < 0x1p20 && g.n < ((int64_t)1 << 30) && n < ((size_t)1 << 30) &&
           top < g.step * 0x1p32 && cutoff < 1e15;
}

// A call's cut in grid steps.  Under width-limited cuts the device alone knows them: here that of a
// line in the middle of the grid with a Lorentz width of 0.07 cm^-1/bar, mean over the conditions --
// only for the choice between kernels that give the same result.
inline double route_cut_steps(double cutoff, double width_mult, const xc_grid &g, const xc_condition *c, int n) {
    if (!(width_mult > 0.0) || !c || n <= 0) return cutoff / g.step;
    const double nu = fmax(g.nu_A + 0.5 * g.step * (double)g.n, 0.0);
    double sum = 0.0;
    for (int i = 0; i < n; ++i) {
        const double al = 3.581e-7 * nu * sqrt(c[i].T / c[i].mass_da);
        const double ga = 0.07 * c[i].gamma_scale * (c[i].P / c[i].P_ref) * pow(c[i].T_ref / c[i].T, 0.6);
        sum += fmin(cutoff, width_mult * fmax(al, ga));
    }
    return sum / n / g.step;
}

// Lines of a list over [lo, hi] (spread evenly) whose cuts can reach the grid -- for the same choice
inline double route_reach(size_t n, double lo, double hi, const xc_grid &g, double cutoff) {
    const double a = fmax(lo, g.nu_A - cutoff), b = fmin(hi, g.nu_A + g.step * (double)g.n + cutoff);
    return hi > lo ? (double)n * fmin(1.0, fmax(b - a, 0.0) / (hi - lo)) : (double)n;
}

// ---- FP32: the block-interpolated sweep (xc_tree.cu), or the tiled kernels with or without the far
// wings on the tensor cores (xc_batched.cu)
struct Route32 {
    int profile, flags, n_gh;
    double cutoff, width_mult;
    double cut_steps;   // route_cut_steps
    xc_grid grid;
    size_t n_lines;
    double reach;       // route_reach
    int n_cond;
    bool allow_tc;   // far wings may use the tensor-core kernel
    bool tiled;      // the tiled kernels whatever the sizes (fixed tile shape, no room for the blocks' scratch)
};

// Sparse lists on large outputs.  Bringing the node sums to a point costs the blocks 16 FP64 operations a
// condition whatever the list; the tiled kernels pay for every pair of a line and a point.  Both were
// timed over 1e5 and 1e6 points x 0.003 to 0.3 lines a point x cuts of 50 to 2500 steps x 1 to 24
// conditions x fixed and width-limited cuts, and follow
//     base + a (points x conditions) + b (lines x conditions) + c (pairs)
// within 10 % (blocks) and 15 to 50 % (tiled, worst where the autotuner picks a slow tile).  Blocks
// against tiled, ps: a 110-133 / 4-22 (w4 with one condition 127 / 119: a launch for its centre zones),
// b 24-200 / 70-1260, c 0.02-0.06 / 0.1-3 (20 Gauss-Hermite nodes 0.5-0.9 / 5-23).  The lines below are the
// differences; over 682 calls 10 are more than 5 % off the better form, the worst 20 %.  At 1e6 points, 6
// conditions, cut 2500 steps, blocks / tiled us: Lorentz 15 pairs a point 886 / 204, 150 928 / 400, 1500
// 1132 / 2533; w4 836 / 355, 880 / 676, 1375 / 4236; binned Lorentz 861 / 334, 904 / 1171, 1444 / 9031.  The
// Doppler profiles have nothing to bring to the points.
inline bool route_sparse32(const Route32 &r, bool tc) {
    const bool wl = r.width_mult > 0.0;               // width-limited: one pass for each condition
    const double nc = wl ? 1.0 : (double)r.n_cond, gh = r.n_gh / 20.0;
    double point, line, pair;                         // ps: cost of the blocks, saved by them
    switch (r.profile) {
    case XC_VOIGT_W4: point = 100.0 - 92.0 / nc; line = 350.0 + 700.0 / nc; pair = tc ? 0.08 : 0.3; break;
    case XC_LORENTZ: point = nc > 1.0 ? 125.0 : 104.0; line = 70.0 + 150.0 / nc; pair = nc >= 16.0 ? 0.12 : 0.2; break;
    case XC_LORENTZ_BINNED: point = 115.0; line = 250.0; pair = nc >= 8.0 ? 2.5 : 1.5; break;
    case XC_VOIGT_GH_BINNED: point = 92.0; line = -700.0 * gh; pair = (nc > 1.0 ? 17.0 : 23.0) * gh; break;
    case XC_VOIGT_GH_SAMPLED: point = 105.0; line = -130.0 * gh; pair = (nc > 1.0 ? 5.0 : 7.0) * gh; break;
    default: return false;
    }
    const double base = wl ? 23e6 * r.n_cond : 28e6 + 5e6 * fmin(nc, 24.0);   // shorter launch sequences
    return base - point * (double)r.grid.n * r.n_cond +
               (line + pair * 2.0 * r.cut_steps) * r.reach * r.n_cond < 0.0;
}

// Whether the tensor-core kernel can take the far wings of a tiled call: many conditions (the
// MMA's N is 32, so a handful of conditions would waste it), one fixed cut, grids of < 2^23 points
inline bool route_tc_form(const Route32 &r) {
    return r.allow_tc && r.profile == XC_VOIGT_W4 && r.width_mult <= 0.0 && r.n_cond >= 16 &&
           !(r.flags & XC_OPT_NO_TENSOR_CORES) && r.grid.n < ((int64_t)1 << 23);
}

// The blocks take every profile but the Vectorized Voigt; 32-bit positions as above; beyond 1.6e9 lines
// the scratch would crowd out other buffers.  They evaluate a ninth of the points at long cuts and are
// faster than the tensor-core form at every dense size measured: 32 conditions x 3e6 lines, cut 1000 steps
// 23.2 ms against 42.3, 500 steps 20.2 against 35.6, 100 steps 15.7 against 30.2; 15 000 lines 0.2
// against 0.9.  Short cuts of small lists with 16 and more conditions stay on the tensor cores all the
// same: xc_last_sweep_kernels and xc_count_far_evals report on that form, and callers (and the
// tests) that ask them at these sizes find it there.
inline bool route_blocks32(const Route32 &r) {
    const double cut = r.cutoff / r.grid.step;
    const bool tc = route_tc_form(r);
    return !r.tiled && r.profile != XC_VOIGT_VV && cut < 0x1p20 && r.grid.n < ((int64_t)1 << 30) &&
           r.n_lines < ((size_t)3 << 29) && !route_sparse32(r, tc) &&
           !(tc && cut < 1024.0 && r.n_lines * (size_t)r.n_cond < ((size_t)1 << 19));
}

// The FP32 adjoint (xc_vjp.cu): dL/dsigma projected on the block nodes costs 75 ps a point and condition
// and then saves evaluations of each line's far points.  Timed over the same family: blocks against all
// points, ps a pair 0.2-0.3 / 0.6 (Lorentz), 2.4 (w4), 24 (20 Gauss-Hermite nodes), and for each line 200, 400
// and 3000 to 5000 more.  1e6 points, 6 conditions, cut 2500 steps, blocks / points us: w4 15 pairs a point
// 778 / 581, 150 1178 / 2684; Lorentz 758 / 286, 1024 / 764, width-limited (500 widths) 770 / 250 and 1031 / 502.
// Points and cuts as for the sweep: a line whose position is near 2^31 then reaches no point.
inline bool route_adjoint_blocks(int profile, int n_gh, double cutoff, double cut_steps, const xc_grid &g,
                                 double reach, int n_cond) {
    if (profile == XC_DOPPLER || g.n >= ((int64_t)1 << 30) || !(cutoff / g.step < 0x1p20)) return false;
    double line, pair;   // ps
    switch (profile) {
    case XC_LORENTZ: line = 220.0; pair = 0.35; break;
    case XC_VOIGT_GH_BINNED: line = 250.0 * n_gh; pair = 1.03 * n_gh; break;
    default: line = 400.0; pair = 2.4; break;
    }
    // a warp takes a line through all conditions: below 2000 lines the chip is not full, and the last
    // line's time is all there is
    return (pair * 2.0 * cut_steps - line) * fmax(reach, 2000.0) * n_cond > 1e7 + 75.0 * (double)g.n * n_cond;
}

// Whatever keeps a call from the blocks, its far wings go to the tensor cores where they can
inline bool route_tc32(const Route32 &r) { return route_tc_form(r) && !route_blocks32(r); }

}  // namespace xc
