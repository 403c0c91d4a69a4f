"""The fixed-point collision of the FP64 form has no error of fixed sign: the
mean over many states of the error of a cell's mass and momentum (built for
the host, against long double).

Bound: a population's error is at most a few 1e-18 (rms 4e-18, its rounding to
FP64 for the most part), so a cell's mass or momentum errs by sqrt(19) 4e-18 =
1.7e-17 and the mean of 400 000 of them by 2.8e-20; six times that is 1.7e-19.
The products' rounding constants are means over random low bits and good to
2^-31 of a unit of 8.7e-19.  2e-19 holds both.  (The quadratic part's weights
are 1/8 and 1/4 exactly in the collision, and here.)"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include "fslbm_fixed.cuh"
using namespace fsl;
typedef long double L;
int main(int, char** arg) {
  const double tau = atof(arg[1]), magic = atof(arg[2]), amp = atof(arg[3]), noise = atof(arg[4]), u0 = atof(arg[5]);
  const double gx = atof(arg[6]);
  Par p;
  std::memset(&p, 0, sizeof p);
  p.lam_p = -1.0 / tau;
  p.lam_m = -1.0 / (magic / (tau - 0.5) + 0.5);
  p.inv_lam_m = 1.0 / p.lam_m;
  p.g[0] = gx;
  p.g[2] = -3.7 * gx;
  fix_constants(p);
  std::mt19937_64 bits(1409);
  auto uniform = [&](double a) { return a * (2.0 * (double)(bits() >> 11) * 0x1p-53 - 1.0); };
  L mean[4] = {0, 0, 0, 0};
  int taken = 0;
  for (int n = 0; n < 400000; ++n) {
    const double u[3] = {u0 + uniform(amp), uniform(amp), uniform(amp)}, rho0 = 1.0 + uniform(0.03);
    const double us = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    double f[19], g[19];
    L rho = 0, j[3] = {0, 0, 0};
    for (int q = 0; q < 19; ++q) {
      const double cu = cx(q) * u[0] + cy(q) * u[1] + cz(q) * u[2], w = q == 0 ? 1.0 / 3.0 : (q <= 6 ? 1.0 / 18.0 : 1.0 / 36.0);
      g[q] = f[q] = w * (rho0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * us) * (1.0 + uniform(noise));
      rho += f[q];
      j[0] += cx(q) * (L)f[q];
      j[1] += cy(q) * (L)f[q];
      j[2] += cz(q) * (L)f[q];
    }
    long long r;
    bool fast;
    if (!collide_fixed(p, g, r, fast)) continue;
    ++taken;
    L v[3], usq = 0;  // u^eq, u.u
    for (int a = 0; a < 3; ++a) {
      v[a] = j[a] - (L)p.g[a] / (L)p.lam_m;
      j[a] += (L)p.g[a] / 2;
      usq += j[a] * j[a];
    }
    for (int q = 0; q < 19; ++q) {
      const L w = q == 0 ? 1.0 / 3.0 : (q <= 6 ? 1.0 / 18.0 : 1.0 / 36.0);
      const L cu = cx(q) * j[0] + cy(q) * j[1] + cz(q) * j[2];
      // w (rho - 3/2 u.u) + 9/2 w (c.u)^2
      const L ep = w * (rho - 1.5L * usq) + (q == 0 ? 0.0L : (q <= 6 ? 0.25L : 0.125L)) * cu * cu;
      const L em = (q == 0 ? 0 : q <= 6 ? 2 : 1) * 3.0L * (L)(1.0 / 36.0) * (cx(q) * v[0] + cy(q) * v[1] + cz(q) * v[2]);
      const L want = f[q] + (L)p.lam_p * (((L)f[q] + f[inv(q)]) / 2 - ep) + (L)p.lam_m * (((L)f[q] - f[inv(q)]) / 2 - em);
      const L d = g[q] - want;
      mean[0] += d;
      mean[1] += cx(q) * d;
      mean[2] += cy(q) * d;
      mean[3] += cz(q) * d;
    }
  }
  std::printf("%d", taken);
  for (L m : mean) std::printf(" %.3Le", m / taken);
  std::printf("\n");
}
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("mean")
    (d / "mean.cu").write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "paper_1409_5645_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    str(d / "mean.cu"), "-o", str(d / "mean")], check=True)
    return lambda *a: [float(v) for v in subprocess.run([str(d / "mean"), *map(str, a)], capture_output=True, text=True,
                                                        check=True).stdout.split()]


@pytest.mark.parametrize("tau,magic,amp,noise,u0,gx", [(0.8, 3 / 16, 1e-6, 1e-6, 0.0, 0.0), (0.8, 3 / 16, 1e-6, 1e-6, 0.0, 1e-6),
                                                       (0.55, 3 / 16, 1e-4, 1e-5, 0.0, 2e-5), (0.53, 0.005, 0.04, 0.02, 0.02, 1e-5),
                                                       (1.7, 0.25, 0.05, 0.05, -0.05, 3e-4), (0.51, 3 / 16, 0.05, 0.9, 0.0, 1e-3)])
def test_no_error_of_fixed_sign(driver, tau, magic, amp, noise, u0, gx):
    taken, *mean = driver(tau, magic, amp, noise, u0, gx)
    assert taken > 300000
    assert max(abs(m) for m in mean) < 2e-19, mean
