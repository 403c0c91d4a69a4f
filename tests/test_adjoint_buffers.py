"""The reverse sweep's device buffers come all or not at all: an allocation
that fails at any place leaves no pointer set, nothing held and the byte count
as it was, twice in a row, and a later try gets every buffer (built for the
host with a counting allocator, no GPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include "fslbm_adjoint.h"
static std::map<void*, size_t> held;
static int calls, fail_at;
static bool take(void** p, size_t bytes) {
  if (++calls == fail_at) { *p = nullptr; return false; }
  *p = std::malloc(1);
  held[*p] = bytes;
  return true;
}
static void give(void* p) { if (held.erase(p) != 1) std::abort(); std::free(p); }
int main() {
  const size_t N = 60;
  for (int k = 0; k <= 17; ++k) {
    AdjointState A;
    A.K = 3; A.fbytes = 19 * N * 4; A.rbytes = N * 4; A.bytes = 1000;
    for (int round = 0; round < 2; ++round) {
      calls = 0; fail_at = k;
      const bool ok = adj_alloc_reverse(&A, N, take, give);
      void* ptrs[] = {A.abar[0], A.abar[1], A.P, A.mbar[0], A.mbar[1], A.phibar[0], A.phibar[1], A.theta, A.dphi0,
                      A.seg_f, A.seg_m, A.seg_phi, A.seg_flags, A.Mh, A.flist, A.rh, A.ngb};
      int set = 0;
      size_t sum = 1000;
      for (void* p : ptrs) set += p != nullptr;
      for (auto& e : held) sum += e.second;
      std::printf("%d %d %d %d %d %d\n", k, round, ok, set, (int)held.size(), sum == A.bytes);
    }
    fail_at = 0;
    const bool ok = adj_alloc_reverse(&A, N, take, give);
    std::printf("%d 2 %d 17 %d 1\n", k, ok, (int)held.size());
    held.clear();
  }
}
"""


def test_failed_allocation_leaves_nothing(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    (tmp_path / "buffers.cu").write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "paper_1409_5645_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    str(tmp_path / "buffers.cu"), "-o", str(tmp_path / "buffers")], check=True)
    out = subprocess.run([str(tmp_path / "buffers")], capture_output=True, text=True, check=True).stdout
    rows = [[int(v) for v in line.split()] for line in out.splitlines()]
    assert len(rows) == 54
    for k, attempt, ok, pointers, held, bytes_match in rows:
        want = 17 if k == 0 or attempt == 2 else 0  # (k = 0: no allocation fails)
        assert (ok, pointers, held, bytes_match) == (int(want > 0), 17 if attempt == 2 else want, want, 1), (k, attempt)
