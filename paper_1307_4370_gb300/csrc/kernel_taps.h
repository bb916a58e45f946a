// The interpolation kernels of G (§5) on the host, in double: their values, their
// transforms and the tap weights of the set-up.  Plain C++ (no CUDA), so that
// they can be checked on a host without a GPU.
#pragma once
#include <algorithm>
#include <cmath>

#include "purify.h"

namespace purify {

constexpr int kTapsMaxJ = 8;  // largest kernel support

// ---------------------------------------------------------------------------
// Kaiser-Bessel: beta of Beatty et al. (2005) for oversampling 2, the kernel
// g(t) = I0(beta sqrt(1 - (2t/J)^2)) / I0(beta) and its closed-form transform.
// ---------------------------------------------------------------------------
inline double kb_beta(int J) {
  const double a = 2.0;
  return M_PI * std::sqrt((J / a) * (J / a) * (a - 0.5) * (a - 0.5) - 0.8);
}

inline double kb_g(double t, int J, double beta, double i0b) {
  const double s = 2.0 * t / J;
  if (std::fabs(s) > 1.0) return 0.0;
  return std::cyl_bessel_i(0.0, beta * std::sqrt(std::max(0.0, 1.0 - s * s))) / i0b;
}

inline double kb_ghat(double f, int J, double beta, double i0b) {
  const double a = std::sqrt(beta * beta - (M_PI * J * f) * (M_PI * J * f));
  return J * std::sinh(a) / (i0b * a);
}

// The paper's Gaussian kernel (§5): g(t) = exp(-b t^2) on |t| <= J/2 with
// b = pi (alpha - 1/2) / (alpha J / 2), alpha = 2 (the width of Greengard &
// Lee 2004 in grid cells); g_hat is the transform of the untruncated Gaussian.
inline double gauss_b(int J) { return M_PI * 1.5 / (2.0 * (J / 2.0)); }
inline double gauss_g(double t, int J) { return std::fabs(t) <= J / 2.0 ? std::exp(-gauss_b(J) * t * t) : 0.0; }
inline double gauss_ghat(double f, int J) {
  const double b = gauss_b(J);
  return std::sqrt(M_PI / b) * std::exp(-M_PI * M_PI * f * f / b);
}

// g and g_hat of the context's kernel.
inline double interp_g(double t, int J, int kernel, double beta, double i0b) {
  return kernel == PURIFY_KERNEL_GAUSS ? gauss_g(t, J) : kb_g(t, J, beta, i0b);
}
inline double interp_ghat(double f, int J, int kernel, double beta, double i0b) {
  return kernel == PURIFY_KERNEL_GAUSS ? gauss_ghat(f, J) : kb_ghat(f, J, beta, i0b);
}

// I0 by its power series sum (z^2 / 4)^k / (k!)^2 (positive terms).
inline long double bessel_i0l(long double z) {
  const long double q = z * z / 4;
  long double term = 1, sum = 1;
  for (int k = 1; term > sum * 1e-22L; ++k) {
    term *= q / ((long double)k * k);
    sum += term;
  }
  return sum;
}

// The taps of the set-up's stencils.  The Gaussian's are evaluated as defined.
// The Kaiser-Bessel ones are Chebyshev interpolants of degree 16 in z = 2x - 1
// with coefficients formed in long double: within 3e-16 of the kernel (the
// library Bessel function in double: 4e-15; coefficients formed in double: 6e-15),
// at a tenth of the time of that function, which was a quarter of the set-up
// at M = 2^21.
struct TapSeries {
  static constexpr int kTerms = 17;
  int J, kernel;
  double c[kTapsMaxJ][kTerms];
};

inline double tap_value(const double* c, double z) {  // Clenshaw's recurrence
  double b1 = 0.0, b2 = 0.0;
  for (int k = TapSeries::kTerms - 1; k >= 1; --k) {
    const double b0 = c[k] + 2.0 * z * b1 - b2;
    b2 = b1;
    b1 = b0;
  }
  return c[0] + z * b1 - b2;
}

inline TapSeries fit_taps(int J, int kernel) {
  constexpr int np = TapSeries::kTerms;
  TapSeries p{};
  p.J = J;
  p.kernel = kernel;
  if (kernel == PURIFY_KERNEL_GAUSS) return p;
  const long double beta = kb_beta(J), i0b = bessel_i0l(beta);
  long double ct[4 * np];  // cos(pi m / (2 np)), one period
  for (int m = 0; m < 4 * np; ++m) ct[m] = std::cos(3.14159265358979323846264338327950288L * m / (2 * np));
  for (int a = 0; a < J; ++a) {
    long double f[np];
    for (int i = 0; i < np; ++i) {
      const long double s = 2 * ((ct[2 * i + 1] + 1) / 2 + J / 2 - 1 - a) / J;
      f[i] = bessel_i0l(beta * std::sqrt(std::max(0.0L, 1 - s * s))) / i0b;
    }
    for (int k = 0; k < np; ++k) {
      long double sum = 0;
      for (int i = 0; i < np; ++i) sum += f[i] * ct[k * (2 * i + 1) % (4 * np)];
      p.c[a][k] = (double)(sum * (k == 0 ? 1 : 2) / np);
    }
  }
  return p;
}

// Weights of the J taps for the fraction x in [0, 1).
inline void tap_weights(const TapSeries& p, double x, double* w) {
  if (p.kernel == PURIFY_KERNEL_GAUSS) {
    for (int a = 0; a < p.J; ++a) w[a] = gauss_g(x + p.J / 2 - 1 - a, p.J);
    return;
  }
  for (int a = 0; a < p.J; ++a) w[a] = tap_value(p.c[a], 2.0 * x - 1.0);
}

}  // namespace purify
