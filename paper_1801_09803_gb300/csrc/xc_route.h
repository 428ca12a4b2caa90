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

// ---- FP32: the block-interpolated sweep (xc_tree.cu), or the tiled kernels with or without the far
// wings on the tensor cores (xc_batched.cu)
struct Route32 {
    int profile, flags;
    double cutoff, width_mult;
    xc_grid grid;
    size_t n_lines;
    int n_cond;
    bool allow_tc;   // far wings may use the tensor-core kernel
    bool tiled;      // the tiled kernels whatever the sizes (fixed tile shape, no room for the blocks' scratch)
};

// Sparse lists on large outputs: few pairs of a line and a point for each point.  Bringing the node
// sums to a point costs 16 FP64 operations a condition whatever the list, 118 ps a point, where
// the tiled kernels need 0.42 ps a pair (0.16 on the tensor cores): 1e6 points, cut 2500 steps, blocks
// against tiled: 6 conditions, 15 / 100 / 300 pairs a point 844/399, 874/613, 917/1102 us; 24
// conditions, 15 / 300 / 1000 pairs 2942/911, 3142/1957, 3708/4656 us.  On small outputs launches
// decide and the blocks are no slower (1e5 points, 6 conditions 188/206 us, 24: 398/376, 405/436).
// Below 256 steps of cut most pairs are near ones, which cost the same in both.
inline bool route_sparse32(const Route32 &r, bool tc) {
    if ((r.profile != XC_VOIGT_W4 && r.profile != XC_LORENTZ) || r.cutoff / r.grid.step < 256.0) return false;
    const double outputs = (double)r.grid.n * (double)r.n_cond;
    const double most = outputs >= 0x1p22 ? (tc ? 500.0 : 200.0) : (outputs >= 0x1p21 ? 50.0 : 0.0);
    return 2.0 * r.cutoff / r.grid.step * (double)r.n_lines < most * (double)r.grid.n;
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

// Whatever keeps a call from the blocks, its far wings go to the tensor cores where they can
inline bool route_tc32(const Route32 &r) { return route_tc_form(r) && !route_blocks32(r); }

}  // namespace xc
