// Colour definitions on the device, FP64 (Sec. 3.4.2).
//
// The observer is this project's piecewise-Gaussian colour matching
// functions (in the functional form of Wyman, Sloan and Shirley, JCGT 2013);
// black bodies are integrated on a 5 nm trapezoid grid from 360 to 830 nm.
// The arithmetic is written with explicit round-to-nearest intrinsics where
// the result feeds an integer decision (star binning), so that no
// multiply-add contraction changes the rounding.
#pragma once

#include <cmath>

#include "bh_internal.cuh"

namespace bh {

// Planck's law up to a constant factor; lambda in nm.
__device__ __forceinline__ double dplanck(double l, double T) {
  const double c2 = 1.4387769e7;  // h c / k, nm K
  double l2 = __dmul_rn(l, l);
  double l5 = __dmul_rn(__dmul_rn(l2, l2), l);
  return __ddiv_rn(1.0, __dmul_rn(l5, expm1(__ddiv_rn(c2, __dmul_rn(l, T)))));
}

// XYZ of a black body; cmf[3*k..] holds the matching functions at 360 + 5k nm.
__device__ __forceinline__ void dblackbody_xyz(const double *cmf, double T, double *xyz) {
  xyz[0] = xyz[1] = xyz[2] = 0.0;
  if (!(T > 0.0)) return;
  for (int k = 0; k < kNLambda; ++k) {
    double l = 360.0 + 5.0 * k;
    double w = (k == 0 || k == kNLambda - 1) ? 2.5 : 5.0;
    double b = __dmul_rn(dplanck(l, T), w);
    xyz[0] = __dadd_rn(xyz[0], __dmul_rn(b, cmf[3 * k + 0]));
    xyz[1] = __dadd_rn(xyz[1], __dmul_rn(b, cmf[3 * k + 1]));
    xyz[2] = __dadd_rn(xyz[2], __dmul_rn(b, cmf[3 * k + 2]));
  }
}

// ---------------------------------------------------------------------------
// Fits of black-body sums
//
// The sums over the wavelengths are smooth in v = 1/T once the exponential
// of one wavelength is taken out, so they are fitted on equal cells of v by
// polynomials through N Chebyshev nodes: one black body per node instead of one
// per use.  What does not depend on the cell is computed once on the host (in
// extended precision) and passed as a kernel parameter.
// ---------------------------------------------------------------------------
template <int N>
struct BlackBodyFit {
  double node[N];                      // Chebyshev nodes on [-1, 1]
  // values at the nodes -> monomial coefficients, as sums of two doubles: their
  // terms cancel to a thousandth
  double inv[N][N], inv_lo[N][N];
  double x[kNLambda];                  // c2 / lambda (K)
  double cmf[3][kNLambda];             // matching functions
  double w[3][kNLambda];               // ... times the trapezoid weight over (lambda / 560 nm)^5
};

#pragma nv_diagnostic push
#pragma nv_diag_suppress 20208  // long double: host code only
template <int N>
const BlackBodyFit<N> &black_body_fit() {
  static const BlackBodyFit<N> fit = [] {
    BlackBodyFit<N> f = {};
    const long double pi = 3.14159265358979323846264338327950288L;
    double mono[N][N] = {};  // mono[j][m]: coefficient of u^m in the Chebyshev polynomial T_j
    mono[0][0] = 1.0;
    mono[1][1] = 1.0;
    for (int j = 2; j < N; ++j)
      for (int m = 0; m < N; ++m) mono[j][m] = (m > 0 ? 2.0 * mono[j - 1][m - 1] : 0.0) - mono[j - 2][m];
    for (int k = 0; k < N; ++k) {
      f.node[k] = (double)cosl(pi * (k + 0.5L) / N);
      for (int m = 0; m < N; ++m) {
        long double s = 0.0L;
        for (int j = 0; j < N; ++j) s += mono[j][m] * (j == 0 ? 1.0L : 2.0L) / N * cosl(j * pi * (k + 0.5L) / N);
        f.inv[m][k] = (double)s;
        f.inv_lo[m][k] = (double)(s - f.inv[m][k]);
      }
    }
    auto lobe = [](double l, double m, double s1, double s2) {
      const double t = (l - m) / (l < m ? s1 : s2);
      return exp(-0.5 * t * t);
    };
    for (int k = 0; k < kNLambda; ++k) {  // the observer
      const double l = 360.0 + 5.0 * k, r = l / 560.0, t = (k == 0 || k == kNLambda - 1 ? 2.5 : 5.0) / (r * r * r * r * r);
      f.x[k] = 1.4387769e7 / l;
      f.cmf[0][k] = 1.056 * lobe(l, 599.8, 37.9, 31.0) + 0.362 * lobe(l, 442.0, 16.0, 26.7) -
                    0.065 * lobe(l, 501.1, 20.4, 26.2);
      f.cmf[1][k] = 0.821 * lobe(l, 568.8, 46.9, 40.5) + 0.286 * lobe(l, 530.9, 16.3, 31.1);
      f.cmf[2][k] = 1.217 * lobe(l, 437.0, 11.8, 36.0) + 0.681 * lobe(l, 459.0, 26.0, 13.8);
      for (int c = 0; c < 3; ++c) f.w[c][k] = t * f.cmf[c][k];
    }
    return f;
  }();
  return fit;
}
#pragma nv_diagnostic pop

// Coefficient m of a fit from the values at the nodes (val[k * stride], read
// past L1: other SMs wrote them), summed with what its roundings lost.
template <int N>
__device__ __forceinline__ double fit_coefficient(const BlackBodyFit<N> &fit, int m, const double *val, int stride) {
  double a = 0.0, err = 0.0;
  for (int k = 0; k < N; ++k) {
    const double f = __ldcg(val + k * stride), p = __dmul_rn(fit.inv[m][k], f), t = __dadd_rn(a, p), z = __dadd_rn(t, -a);
    err += (__dadd_rn(a, -__dadd_rn(t, -z)) + __dadd_rn(p, -z)) + (fma(fit.inv[m][k], f, -p) + fit.inv_lo[m][k] * f);
    a = t;
  }
  return a + err;
}

}  // namespace bh
