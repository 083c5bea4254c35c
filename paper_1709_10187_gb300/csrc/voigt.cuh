// voigt.cuh -- device line-profile functions (Sec. 2.1, Sec. 2.2) in FP64.
//
// dawson_f64: F(x) = int_0^x exp(y^2 - x^2) dy.  |x| < 0.5: its power series
//   F(x) = sum_k (-2)^k x^(2k+1) / (2k+1)!!.  Elsewhere Rybicki's (1989,
//   Computers in Physics 3(2)) series F(x) ~ pi^-1/2 sum_{n odd} e^{-(x-nh)^2}/n,
//   re-centred on the even multiple n0 of h closest to x; here h = 1/4 (aliasing
//   error ~ e^{-(2 pi)^2} ~ 7e-18 relative), 16 odd terms on each side summed
//   from the smallest (the first one left out is e^{-64} ~ 2e-28 of the largest,
//   twelve digits below the sum's last bit).
// calH(a, hi) - calH(a, lo) with
//   calH(a,x) = (sqrt(pi)/2) erf x - (2a/sqrt(pi)) F(x) + a^2 x e^{-x^2}
//   (integral of eq. H_approx); the erf difference is taken from erfc on the
//   side away from line centre.  Neighbouring bins share an edge, so what an
//   edge contributes (VoigtEdge) is computed once.
#pragma once
#include <cuda_runtime.h>

namespace rddmc {

constexpr int kDawsonTerms = 16;  // odd terms of Rybicki's series on each side

// F(|x|) for |x| < 0.5.
__device__ __forceinline__ double dawson_series_f64(double ax) {
    const double x2 = ax * ax;
    double term = ax, sum = ax;
    for (int k = 1; k < 30; ++k) {
        term = term * (-2.0 * x2) / (double)(2 * k + 1);
        sum += term;
        if (fabs(term) < 0x1p-56 * sum) break;  // the terms only get smaller: the sum stays
    }
    return sum;
}

// Terms n' = +m and n' = -m, m = 2 i + 1, of Rybicki's series at |x| >= 0.5.
struct DawsonCentre {
    double n0, xp;  // the even multiple of h = 1/4 closest to |x|, |x| - n0 h
    __device__ __forceinline__ explicit DawsonCentre(double ax) : n0(2.0 * rint(ax / (2.0 * 0.25))), xp(ax - n0 * 0.25) {}
    __device__ __forceinline__ double term(int i) const {
        const double m = (double)(2 * i + 1);
        const double dp = xp - m * 0.25, dm = xp + m * 0.25;
        return exp(-dp * dp) / (n0 + m) + exp(-dm * dm) / (n0 - m);
    }
};
constexpr double kInvSqrtPi = 0.56418958354775628695;

__device__ __forceinline__ double dawson_f64(double x) {
    const double ax = fabs(x);
    double res;
    if (ax < 0.5) {
        res = dawson_series_f64(ax);
    } else {
        const DawsonCentre c(ax);
        double sum = 0.0;
        for (int i = kDawsonTerms - 1; i >= 0; --i) sum += c.term(i);
        res = sum * kInvSqrtPi;
    }
    return x < 0.0 ? -res : res;
}

// What bin edge x contributes to calH differences.
struct VoigtEdge {
    double F;     // Dawson's integral
    double g;     // x e^{-x^2}
    double erfc;  // erfc(|x|)
    double x;
};

__device__ __forceinline__ VoigtEdge voigt_edge(double x, double F) {
    return VoigtEdge{F, x * exp(-x * x), erfc(fabs(x)), x};
}

__device__ __forceinline__ double voigt_hint_diff_f64(double a, const VoigtEdge& lo, const VoigtEdge& hi) {
    double derf;
    if (lo.x >= 0.0)
        derf = lo.erfc - hi.erfc;
    else if (hi.x <= 0.0)
        derf = hi.erfc - lo.erfc;
    else
        derf = erf(hi.x) - erf(lo.x);
    return 0.88622692545275801365 * derf - 2.0 * a * kInvSqrtPi * (hi.F - lo.F) + a * a * (hi.g - lo.g);
}

// Bin mean of H between two edges (k_j / k0 of Sec. 2.2).
__device__ __forceinline__ double voigt_bin_mean_f64(double a, const VoigtEdge& lo, const VoigtEdge& hi) {
    return voigt_hint_diff_f64(a, lo, hi) / (hi.x - lo.x);
}

}  // namespace rddmc
