// acm_roots.h -- the twiddle table of the FP64 transforms (host code, plain C++).
#pragma once
#include <cmath>

namespace acm {

// out[2k], out[2k + 1] = Re, Im of exp(-2 pi i k / n), n a multiple of 8: the first
// octant is evaluated in long double and reflected, so that the values are the
// nearest doubles and the multiples of a quarter turn are exact. Cosine and sine of
// the double nearest to 2 pi k / n are up to 6.5e-16 off at n = 1024, more than the
// arithmetic of a whole transform rounds (relative L2 error of r2c at 64^3: 3.5e-16
// with those, 2.8e-16 with these; FP32 entries are the same either way).
inline void unit_roots(int n, double* out) {
  auto put = [&](int k, double re, double im) {
    out[2 * k] = re;
    out[2 * k + 1] = im;
  };
  for (int k = 0; k <= n / 8; ++k) {
    const long double a = 2.0L * 3.14159265358979323846264338327950288L * k / n;
    const double c = (double)std::cos(a), s = (double)std::sin(a);
    // k and its mirror image about pi / 4, each turned by 0 to 3 quarters
    for (int q = 0; q < 4; ++q) {
      const double re[4] = {c, -s, -c, s}, im[4] = {-s, -c, s, c};
      put(k + q * (n / 4), re[q], im[q]);
      const double re2[4] = {s, -c, -s, c}, im2[4] = {-c, -s, c, s};
      if (k > 0) put(n / 4 - k + q * (n / 4), re2[q], im2[q]);
    }
  }
}

}  // namespace acm
