"""The FP64 twiddle table (csrc/acm_roots.h) against extended precision. CPU only."""
import subprocess

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <vector>
#include "acm_roots.h"
int main() {
  for (int n : {8, 64, 1024}) {
    double worst = 0;
    bool quarters = true;
    std::vector<double> t(2 * n, 7.0);
    acm::unit_roots(n, t.data());
    for (int k = 0; k < n; ++k) {
      const double c = t[2 * k], s = t[2 * k + 1];
      const long double a = 2.0L * 3.14159265358979323846264338327950288L * k / n;
      worst = std::fmax(worst, (double)std::fmax((long double)std::fabs(c - std::cos(a)), (long double)std::fabs(s + std::sin(a))));
      if (k % (n / 4) == 0) quarters = quarters && (c == 0 || s == 0) && c * c + s * s == 1;
    }
    printf("%.3e %d\n", worst, (int)quarters);
  }
  return 0;
}
"""


def test_table_entries_are_the_nearest_doubles(tmp_path):
    from paper_2312_15554_gb300 import build
    src, exe = tmp_path / "r.cpp", tmp_path / "r"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", build.CSRC, str(src), "-o", str(exe)], check=True)
    for line in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")[:3]:
        worst, quarters = line.split()
        # half a unit in the last place of values below 1, and the reference's own rounding
        assert float(worst) <= 0.5 * 2.0 ** -53 * 1.01
        assert quarters == "1"
