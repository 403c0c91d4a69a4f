"""quot_near, the quotients of one divisor by one division, rounds as a
division does (built for the host): divisors of the kernels (1 to 18, a
normal's length and its L1 norm), dividends of every size they have."""
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
