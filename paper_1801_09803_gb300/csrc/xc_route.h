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

}  // namespace xc
