"""Which way steps go out, from the profiler's record of launches: many steps of
a small lattice in one launch only where more than four are asked for and the
kernels are not wanted in order; graphs only where they pay."""
import pytest

from paper_1409_5645_gb300 import cases, fslbm

pytestmark = pytest.mark.gpu


def _record(work):
    """Launches of a call: names of kernels and runtime calls with their counts."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    out = {}
    for _ in range(2):  # (the first profile of a process may come back empty)
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            work()
            torch.cuda.synchronize()
        out = {e.key: e.count for e in p.key_averages()}
        if any("fsl::" in k for k in out):
            return out
    pytest.skip("the profiler records no kernels here")


def _count(record, name):
    return sum(n for k, n in record.items() if name in k)


@pytest.fixture(scope="module", autouse=True)
def _profiler():
    g = fslbm.Lattice.from_case(cases.dam_break(nx=24, ny=8, nz=16, col_x=8, col_z=12, tau=0.6, g=2e-4))
    _record(lambda: g.step(1) or g.sync())


def test_many_steps_launch():
    c = cases.dam_break(nx=24, ny=8, nz=16, col_x=8, col_z=12, tau=0.6, g=2e-4)
    for precision in ("f64", "f32"):
        g = fslbm.Lattice.from_case(c, precision=precision)
        bulk = "k_bulk"
        r = _record(lambda: g.step(20) or g.sync())
        assert _count(r, "k_steps") == 1 and _count(r, bulk) == 1
        r = _record(lambda: g.step(4) or g.sync())
        assert _count(r, "k_steps") == 0 and _count(r, bulk) == 4
        g.set_overlap(False)
        r = _record(lambda: g.step(20) or g.sync())
        assert _count(r, "k_steps") == 0 and _count(r, bulk) == 20
        g.set_overlap(True)
        r = _record(lambda: g.step(20) or g.sync())
        assert _count(r, "k_steps") == 1 and _count(r, bulk) == 1


def test_graphs_where_they_pay():
    """A fresh handle: short calls by kernels, for eight steps at once up to its
    sixteenth such step, for single ones up to its second; a call of sixteen and
    more by graphs at once."""
    c = cases.dam_break(nx=96, ny=32, nz=32, col_x=32, col_z=22, tau=0.6, g=2e-4)
    g = fslbm.Lattice.from_case(c, precision="f32", bulk_loads="pairs")
    # 8: a step by kernels (eight to go), one more, six single graphs; 9: two by kernels, seven single graphs
    for n, launches in ((8, 6), (9, 7), (24, 3), (8, 1), (8, 1)):
        r = _record(lambda: g.step(n) or g.sync())
        assert _count(r, "k_bulk_pairs") == n and _count(r, "cudaGraphLaunch") == launches, n
    g = fslbm.Lattice.from_case(c, precision="f32", bulk_loads="pairs")
    for launches in (0, 0, 1, 1):
        r = _record(lambda: g.step(1) or g.sync())
        assert _count(r, "cudaGraphLaunch") == launches and _count(r, "k_bulk_pairs") == 1
    g = fslbm.Lattice.from_case(c, precision="f32", bulk_loads="pairs")
    r = _record(lambda: g.step(16) or g.sync())
    assert _count(r, "cudaGraphLaunch") == 2 and _count(r, "k_bulk_pairs") == 16
