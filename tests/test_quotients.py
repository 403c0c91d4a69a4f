"""quot_near, the quotients of one divisor by one division, and over_root, a
vector over its length, round as a division and a square root do (built for
the host): divisors of the kernels (1 to 18, a normal's length and its L1
norm), dividends of every size they have, reciprocals off by an ulp too."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "fslbm_dev.cuh"
int main() {
  std::mt19937_64 bits(3);
  auto u = [&]() { return (double)(bits() >> 11) * 0x1p-53; };
  long long bad = 0;
  for (int n = 0; n < 3000000; ++n) {
    const double b = n % 3 == 0 ? 1.0 + (double)(bits() % 18) : (n % 3 == 1 ? 1.0 + u() : std::exp(20.0 * (u() - 0.9)));
    const double a = (u() - 0.5) * std::exp(12.0 * (u() - 0.5)) * (n % 7 ? 1.0 : b);
    bad += fsl::quot_near(a, b, 1.0 / b) != a / b;
  }
  bad += fsl::quot_near(0.0, 3.0, 1.0 / 3.0) != 0.0;
  for (int n = 0; n < 1000000; ++n) {
    const double scale = std::exp(24.0 * (u() - 0.95));
    const double v[3] = {(u() - 0.5) * scale, (u() - 0.5) * scale, n % 5 ? (u() - 0.5) * scale : 0.0};
    const double s = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
    double w[3] = {v[0], v[1], v[2]};
    fsl::over_root<false>(w[0], w[1], w[2], s);
    for (int a = 0; a < 3; ++a) {
      bad += w[a] != v[a] / std::sqrt(s);
      const double y = std::nextafter(1.0 / std::sqrt(s), n % 2 ? 0.0 : 1e300);  // (as rsqrt may be)
      const double t = s * y, len = fma(fma(-t, t, s), 0.5 * y, t);
      bad += len != std::sqrt(s) || fsl::quot_near(v[a], len, y) != v[a] / len;
    }
  }
  std::printf("%lld\n", bad);
}
"""


def test_as_a_division(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    (tmp_path / "quot.cu").write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "paper_1409_5645_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    str(tmp_path / "quot.cu"), "-o", str(tmp_path / "quot")], check=True)
    assert int(subprocess.run([str(tmp_path / "quot")], capture_output=True, text=True, check=True).stdout) == 0
