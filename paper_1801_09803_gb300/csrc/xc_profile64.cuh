// xc_profile64.cuh -- the FP64 line profiles (unit area) at offset D from the centre.
#pragma once

#include "xc_internal.cuh"

namespace xc {

template <int PROF>
__device__ inline double profile64(double D, double step, double al, double ga, const double *ghx,
                                   const double *ghw, int ngh, double nul = 0.0, double split = 4.0,
                                   int beta = 0) {
    if (PROF == XC_VOIGT_VV) {
        return voigt_vv64(D, al, ga, nul, split, beta);
    } else if (PROF == XC_DOPPLER) {
        // Eq. (e:Gauss): sqrt(ln2/pi)/alpha exp(-D^2 ln2/alpha^2)
        double r = D / al;
        return 0.46971863934982566 / al * exp(-kLn2 * r * r);
    } else if (PROF == XC_LORENTZ) {
        // Eq. (e:lor)
        return ga / (kPi * (D * D + ga * ga));
    } else if (PROF == XC_VOIGT_W4) {
        // unit-area Voigt: sqrt(ln2/pi)/alpha Re w(x + iy), x = sqrt(ln2) D/alpha, y = sqrt(ln2) gamma/alpha
        double ia = kSqrtLn2 / al;
        Cx<double> w = w4_eval<double>(D * ia, ga * ia, nullptr);
        return 0.46971863934982566 / al * w.re;
    } else if (PROF == XC_DOPPLER_BINNED) {
        // Eq. (eqn:sig_ij) without I: (erf(x+) - erf(x-)) / (2h), x+- = sqrt(ln2)/alpha (D +- h/2),
        // taken on the side |D| as erfc(x-) - erfc(x+) (the profile is symmetric)
        double t = fabs(D), c = kSqrtLn2 / al;
        return (erfc(c * (t - 0.5 * step)) - erfc(c * (t + 0.5 * step))) / (2.0 * step);
    } else if (PROF == XC_LORENTZ_BINNED) {
        // Eq. (eqn:sig_lor-2) without I: (atan(y+) - atan(y-)) / (pi h), y+- = (D +- h/2)/gamma,
        // as one atan2 with both arguments scaled by gamma^2 > 0
        double hh = 0.5 * step;
        return atan2(step * ga, (D + hh) * (D - hh) + ga * ga) / (kPi * step);
    } else if (PROF == XC_VOIGT_GH_SAMPLED) {
        // Eq. (e:V-quad) with node shift alpha x_j / sqrt(ln2)
        double s = 0.0, g2 = ga * ga, sh = al / kSqrtLn2;
        for (int j = 0; j < ngh; ++j) {
            double d = D - sh * ghx[j];
            s += ghw[j] * ga / (d * d + g2);
        }
        return s * 0.17958712212516656;  // pi^(-3/2)
    } else {
        // Eq. (e:sigma:quad) without I: pi^(-3/2)/h sum_j w_j [atan(y+) - atan(y-)],
        // with atan(a) - atan(b) = atan2(a - b, 1 + ab) for a > b
        double s = 0.0, sh = al / kSqrtLn2, hh = 0.5 * step;
        for (int j = 0; j < ngh; ++j) {
            double d = D - sh * ghx[j];
            double q = (d + hh) * (d - hh) + ga * ga;  // gamma^2 (1 + y+ y-)
            s += ghw[j] * atan2(step * ga, q);          // scaled by gamma^2 > 0 in both arguments
        }
        return s * 0.17958712212516656 / step;
    }
}

}  // namespace xc
