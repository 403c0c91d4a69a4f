"""The bench's roofline notes: a committed profile counts for a kernel only
while the files that kernel is built from stay as they were, and no other
file's change touches it."""
import importlib.util
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def bench():
    spec = importlib.util.spec_from_file_location("bench_module", os.path.join(ROOT, "bench.py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    return m


def test_sources_of_each_bulk_kernel(bench):
    for form, own in (("f64", "fslbm_bulk64.cu"), ("f32", "fslbm_pairs.cu"), ("f16", "fslbm_pairs.cu")):
        names = {os.path.basename(f) for f in bench.kernel_sources(form)}
        assert {own, "fslbm_dev.cuh", "fslbm_pull.cuh", "fslbm_slow.cuh", "fslbm_fixed.cuh"} == names


def test_profiles_belong_to_the_present_kernels(bench):
    for form in ("f64", "f32", "f16"):
        text = open(os.path.join(ROOT, "profiles", f"k_bulk_dam_break_{form}.md")).read()
        assert re.search(r"kernel_source_sha:\s*([0-9a-f]+)", text).group(1) == bench.kernel_source_sha(form)
    assert bench.ncu_traffic("f32") > 1e9 and bench.ncu_traffic("f16") > 5e8
    assert bench.profile_number("f64", "integer_instructions_per_liquid_cell") > 100


def test_no_fp64_rate_bound_in_the_line(bench):
    """The FP64 bulk kernel collides in integers: its line holds no share of the FP64 rate."""
    assert not hasattr(bench, "fp64_counts_per_cell")
    assert "fp64_rate(" not in open(os.path.join(ROOT, "bench.py")).read()
