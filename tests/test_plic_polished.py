"""The FP64 inverse of the plane/unit-cube volume (plic_alpha_polished): its
root against a bisection in extended precision, over random, nearly flat and
degenerate normals and the ends of every range (built for the host, no GPU).
The inverse errs by a few FP64 roundings of numbers below 1/2, so 1e-15."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
LD = np.longdouble
SOURCE = """
#include <cstdio>
#include "fslbm_dev.cuh"
int main() {
  double tv, m1, m2, m3;
  while (std::scanf("%lf %lf %lf %lf", &tv, &m1, &m2, &m3) == 4)
    std::printf("%.17g\\n", fsl::plic_alpha_polished(tv, m1, m2, m3));
}
"""


def volume(a, m1, m2, m3):
    if a <= 0:
        return LD(0)
    if a <= m1:
        return a ** 3 / (6 * m1 * m2 * m3)
    base, den, m12 = 3 * a * a - 3 * a * m1 + m1 * m1, 6 * m2 * m3, m1 + m2
    if a <= m2:
        return base / den
    base = base - (a - m2) ** 3 / max(m1, LD(1e-300))
    if m3 >= m12:
        return base / den if a <= m12 else (a - m12 / 2) / m3
    if a <= m3:
        return base / den
    return (3 * a * a - 3 * a * m1 + m1 * m1 - (a - m2) ** 3 / m1 - (a - m3) ** 3 / m1) / den


def root(tv, *m):
    lo, hi, m = LD(0), LD(0.5), [LD(v) for v in m]
    for _ in range(75):
        mid = (lo + hi) / 2
        lo, hi = (mid, hi) if volume(mid, *m) < LD(tv) else (lo, mid)
    return (lo + hi) / 2


def rows():
    rng = np.random.default_rng(7)
    out = []
    for k in range(1500):
        m = {0: rng.random(3), 1: 10.0 ** rng.uniform(-17, 0, 3), 2: 1 / 3 + 1e-3 * rng.standard_normal(3),
             3: np.array([10.0 ** rng.uniform(-9, -1), rng.random(), rng.random()])}[k % 4]
        m = np.sort(m) / m.sum()
        out.append((max(rng.random() * 0.5 if k % 3 else 0.5 * 10.0 ** rng.uniform(-8.6, 0), 1e-9), *m))
        for a in (m[0], m[1], min(m[0] + m[1], m[2], 0.5)):  # the ends of the ranges
            tv = float(volume(LD(a), *(LD(v) for v in m))) if m[0] > 0 else 0.1
            out.append((min(max(tv, 1e-9), 0.5), *m))
    for m in ([0, 0, 1], [0, 0.3, 0.7], [0, 0.5, 0.5], [0.25, 0.25, 0.5], [0.2, 0.3, 0.5], [1e-40, 0.4, 0.6]):
        out += [(tv, *m) for tv in (1e-9, 1e-6, 0.1, 0.25, 0.5)]
    return out


def test_polished_root(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "polished.cu", str(tmp_path / "polished")
    src.write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "paper_1409_5645_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    str(src), "-o", exe], check=True)
    cells = rows()
    text = "\n".join("%.17g %.17g %.17g %.17g" % c for c in cells)
    got = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split()
    worst = max(float(abs(LD(float(g)) - root(*c))) for g, c in zip(got, cells))
    assert len(got) == len(cells) and worst < 1e-15, worst
