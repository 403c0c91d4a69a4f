"""The fixed-point collision leaves densities far from 1 to collide<double>: a
density of zero is reported there, and a small one keeps its relative
precision (the fixed-point unit is absolute)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1409_5645_gb300 import cases

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <cstdio>
#include <cstring>
#include "fslbm_fixed.cuh"
using namespace fsl;
int main() {
  Par p;
  std::memset(&p, 0, sizeof p);
  p.lam_p = p.lam_m = -1.25;
  p.inv_lam_m = -0.8;
  fix_constants(p);
  double rho;
  while (std::scanf("%lf", &rho) == 1) {
    double f[19];
    for (int q = 0; q < 19; ++q) f[q] = rho * (q == 0 ? 1.0 / 3.0 : (q <= 6 ? 1.0 / 18.0 : 1.0 / 36.0));
    long long r;
    bool fast;
    std::printf("%d\n", collide_fixed(p, f, r, fast));
  }
}
"""


def test_densities_taken(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    (tmp_path / "d.cu").write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "paper_1409_5645_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    str(tmp_path / "d.cu"), "-o", str(tmp_path / "d")], check=True)
    rhos = [0.0, 1e-300, 1e-6, 0.1, 0.49, 0.51, 0.9, 1.0, 1.99, 2.01, 2.9]
    out = subprocess.run([str(tmp_path / "d")], input=" ".join(map(str, rhos)), capture_output=True, text=True, check=True)
    assert [bool(int(v)) for v in out.stdout.split()] == [0.5 <= r < 2 for r in rhos]


def _box(rho):
    dims = (16, 8, 8)
    N = 1024
    return (dims, cases.default_params(tau=0.8, periodic=(1, 1, 1)), np.full(N, cases.LIQUID, np.uint8), rho,
            np.zeros((N, 3)), np.zeros(N))


@pytest.mark.gpu
@pytest.mark.parametrize("steps", [1, 6])  # by the step's kernels, and many in one launch
def test_zero_density_is_refused(steps):
    from paper_1409_5645_gb300 import fslbm
    rho = np.ones(1024)
    rho[500:] = 0.0  # (cells whose neighbours are empty too)
    dims, params, flags, rho, u, phi = _box(rho)
    g = fslbm.Lattice(dims, params)
    g.init_equilibrium(flags, rho, u, phi)
    with pytest.raises(fslbm.FslbmError) as e:
        g.step(steps)
        g.sync()
    assert e.value.code == -5 and "density" in str(e.value)


@pytest.mark.gpu
@pytest.mark.parametrize("steps", [1, 6])
def test_relative_precision_of_small_densities(steps):
    """At rest the collision is linear, so FP64 gives a state scaled by a power
    of two the scaled bits."""
    from paper_1409_5645_gb300 import fslbm
    fields = []
    for scale in (1.0, 2.0 ** -20):
        dims, params, flags, rho, u, phi = _box(np.full(1024, 0.374 * scale))
        g = fslbm.Lattice(dims, params)
        g.init_equilibrium(flags, rho, u, phi)
        g.step(steps)
        fields.append(g.get(fslbm.FIELD_F | fslbm.FIELD_RHO))
    for k in ("f", "rho"):
        assert np.array_equal(fields[0][k] * 2.0 ** -20, fields[1][k]), k
