"""The fixed-point collision of the FP64 form (collide_fixed) on the host
against exact rationals with the FP64 weights: its error bound over states of
a flow, and the states that it must leave to collide<double>.

Bound: a population's result is x + P + M with P, M products in units of
2^-60.  Each product errs by at most 1.25 units itself and carries its
operand's error (at most 2 |lambda| times: e^+ holds a density product and
shifts of products, about 4 units; twice that for the rest population), so
with |lambda| < 2 about 25 units, 2.2e-17, before the rounding to FP64 (half
a spacing, 2.8e-17 for the rest population, 3.5e-18 to 7e-18 for the others):
5.1e-17.  The dropped bits of populations below 2^-8 add one unit each to the
density.  1e-16 holds all of it."""
import os
import random
import shutil
import struct
import subprocess
from fractions import Fraction as F

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <cstdio>
#include <cstring>
#include <cmath>
#include "fslbm_fixed.cuh"
using namespace fsl;
int main() {
  double tau, magic, g[3], f[19];
  while (std::scanf("%lf %lf %lf %lf %lf", &tau, &magic, g, g + 1, g + 2) == 5) {
    for (double& v : f) std::scanf("%lf", &v);
    Par p;
    std::memset(&p, 0, sizeof p);
    p.lam_p = -1.0 / tau;
    p.lam_m = -1.0 / (magic / (tau - 0.5) + 0.5);
    p.inv_lam_m = 1.0 / p.lam_m;
    p.fix_ok = 1;
    p.fx_lp = std::llround(p.lam_p * 0x1p62);
    p.fx_lm = std::llround(p.lam_m * 0x1p62);
    for (int a = 0; a < 3; ++a) {
      p.fx_hg[a] = std::llround(g[a] * 0x1p59);
      p.fx_gl[a] = std::llround(g[a] * p.inv_lam_m * 0x1p60);
    }
    p.fx_um2 = std::llround(0.16 * 0x1p60);
    long long rho = 0;
    bool fast = false;
    const bool ok = collide_fixed(p, f, rho, fast);
    std::printf("%d %d %.17g", ok, fast, double_of_fix(rho));
    for (double v : f) std::printf(" %.17g", v);
    std::printf(" %.17g %.17g\n", p.lam_p, p.lam_m);
  }
}
"""
C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
     (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
     (0, -1, 1)]
W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("fixed")
    (d / "fixed.cu").write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "paper_1409_5645_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    str(d / "fixed.cu"), "-o", str(d / "fixed")], check=True)

    def run(rows):
        text = "\n".join(" ".join("%.17g" % v for v in (r[0], r[1], *r[2], *r[3])) for r in rows)
        out = subprocess.run([str(d / "fixed")], input=text, capture_output=True, text=True, check=True).stdout
        return [[float(v) for v in line.split()] for line in out.splitlines()]

    return run


def state(rng, amp, noise):
    u, rho = [rng.uniform(-amp, amp) for _ in range(3)], rng.uniform(0.97, 1.03)
    usq = sum(v * v for v in u)
    f = []
    for q in range(19):
        cu = sum(a * b for a, b in zip(C[q], u))
        f.append(W[q] * (rho + 3 * cu + 4.5 * cu * cu - 1.5 * usq) * (1 + rng.uniform(-noise, noise)))
    return f


def collide(lp, lm, g, f):
    f, lp, lm, g = [F(v) for v in f], F(lp), F(lm), [F(v) for v in g]
    rho, j = sum(f), [sum(C[q][a] * f[q] for q in range(19)) for a in range(3)]
    u, v = [j[a] + g[a] / 2 for a in range(3)], [j[a] - g[a] / lm for a in range(3)]
    usq, out = sum(x * x for x in u), []
    for q in range(19):
        b, w = (0 if q == 0 else (q + 1 if q % 2 else q - 1)), F(W[q])
        cu, cv = sum(c * x for c, x in zip(C[q], u)), sum(c * x for c, x in zip(C[q], v))
        ep = w * (rho + F(3, 2) * (3 * cu * cu - usq))
        out.append(f[q] + lp * ((f[q] + f[b]) / 2 - ep) + lm * ((f[q] - f[b]) / 2 - 3 * w * cv))
    return out, rho, usq


@pytest.mark.parametrize("tau,magic,amp,noise", [(0.53, 0.005, 0.1, 0.02), (0.8, 3 / 16, 1e-6, 1e-6), (1.7, 0.25, 0.2, 0.1),
                                                 (0.51, 3 / 16, 0.05, 0.9)])
def test_error_bound(driver, tau, magic, amp, noise):
    rng = random.Random(1409)
    rows = [(tau, magic, (1e-5, -2e-4, rng.uniform(-4e-3, 4e-3)), state(rng, amp, noise)) for _ in range(200)]
    taken = 0
    for (t, m, g, f), got in zip(rows, driver(rows)):
        if not got[0]:
            continue
        taken += 1
        want, rho, usq = collide(got[22], got[23], g, f)
        assert max(abs(float(F(a) - b)) for a, b in zip(got[3:22], want)) < 1e-16
        assert abs(float(F(got[2]) - rho)) < 2.3e-16  # (printed in FP64)
        assert bool(got[1]) == (usq > F(16, 100))
    assert taken > 150


def test_out_of_range_states_are_left_alone(driver):
    rng = random.Random(3)
    base = state(rng, 0.05, 0.01)
    bad = []
    for q, v in ((3, -1e-3), (0, 1.0), (7, 0.25), (5, float("nan")), (9, float("inf")), (0, -0.2), (12, -0.0)):
        f = list(base)
        f[q] = v
        bad.append(f)
    bad.append([v * 5 for v in base])                                # a density of 5
    fast = [0.24 if C[q][0] > 0 else 1e-3 for q in range(19)]          # a momentum above 1/2
    bad.append(fast)
    rows = [(0.8, 3 / 16, (0.0, 0.0, 0.0), f) for f in bad]
    for (_, _, _, f), got in zip(rows, driver(rows)):
        assert got[0] == 0
        assert [struct.pack("d", v) for v in got[3:22]] == [struct.pack("d", v) for v in f] or any(v != v for v in f)
    # tiny and zero populations are in range; a negative result takes the general conversion
    for f in ([0.3] + [1e-9] * 6 + [0.05] * 12, [0.3] + [0.0] * 6 + [0.05] * 12, [0.9] + [1e-4] * 18):
        (got,) = driver([(0.55, 3 / 16, (0.0, 0.0, 0.0), f)])
        want, _, _ = collide(got[22], got[23], (0.0, 0.0, 0.0), f)
        assert got[0] == 1 and max(abs(float(F(a) - b)) for a, b in zip(got[3:22], want)) < 1.2e-16
