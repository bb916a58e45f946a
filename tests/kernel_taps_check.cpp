// Host check of the set-up's tap weights (csrc/kernel_taps.h), no GPU needed:
// against the kernels' definitions in long double (I0 by its power series) at
// float32 fractions, as the device stores them.
//
// usage: kernel_taps_check J kernel   (prints "ok <largest error>" or the failure)
#include <cmath>
#include <cstdio>
#include <cstdlib>

#include "kernel_taps.h"

using namespace purify;

static long double i0(long double z) {
  long double term = 1, sum = 1;
  for (int k = 1; k < 200; ++k) {
    term *= z * z / 4 / ((long double)k * k);
    sum += term;
  }
  return sum;
}

int main(int argc, char** argv) {
  if (argc != 3) return 2;
  const int J = std::atoi(argv[1]), kernel = std::atoi(argv[2]);
  const TapSeries taps = fit_taps(J, kernel);
  const long double beta = kb_beta(J), b = gauss_b(J);
  double worst = 0;
  for (int i = 0; i < 6000; ++i) {
    const float x = i < 3 ? (i == 0 ? 0.f : i == 1 ? 1e-7f : std::nextafter(1.f, 0.f)) : (float)((i + 0.37) / 6000.0);
    double w[kTapsMaxJ];
    tap_weights(taps, x, w);
    for (int a = 0; a < J; ++a) {
      const long double t = (long double)x + J / 2 - 1 - a, s = 2 * t / J;
      const long double want =
          kernel == PURIFY_KERNEL_GAUSS ? std::exp(-b * t * t) : i0(beta * std::sqrt(1 - s * s)) / i0(beta);
      worst = std::fmax(worst, (double)std::fabs(w[a] - want));
    }
  }
  // values of at most 1, a sum of 17 terms or an exponential of an argument
  // rounded twice: eight units of rounding
  if (!(worst <= 8 * 1.1102230246251565e-16)) {
    std::printf("FAIL %.3e\n", worst);
    return 1;
  }
  std::printf("ok %.3e\n", worst);
  return 0;
}
