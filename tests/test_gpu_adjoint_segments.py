"""The forward window of a differentiation is the same whatever its
checkpoint distance: the segments go out as many steps in one launch, as graphs or
kernel by kernel, and the recomputation in the reverse sweep once more by
its own rule; with conversions inside, the states are the same bits."""
import numpy as np
import pytest

from paper_1409_5645_gb300 import cases, fslbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rule", [0, 1])
@pytest.mark.parametrize("precision", ["f64", "f32", "f16"])
def test_segments_do_not_show(precision, rule):
    """K = 40: one launch of 39 steps and one by kernels; K = 3 and 1: every
    step by kernels (forward), segments of 2 + 1 in the reverse sweep."""
    c = cases.dam_break(nx=24, ny=8, nz=16, col_x=8, col_z=12, tau=0.6, g=2e-4, rule=rule)
    ref = None
    for K in (40, 3, 1):
        g = fslbm.Lattice.from_case(c, precision=precision, keep_f0=1)
        J = g.adjoint_forward(40, K)
        state = g.get(63)
        dnu, dg, dphi = g.adjoint_backward()
        if ref is None:
            ref = J, state, dnu, dg, dphi
            assert (state["flags"] != c["flags"]).any()
            continue
        for k in state:
            assert np.array_equal(state[k], ref[1][k]), (K, k)
        assert J == ref[0]
        # (the reverse sweep adds some adjoints by atomics, in any order)
        assert dnu == pytest.approx(ref[2], rel=1e-11)
        assert np.abs(dg - ref[3]).max() <= 1e-11 * np.abs(ref[3]).max()
        assert np.abs(dphi - ref[4]).max() <= 1e-11 * np.abs(ref[4]).max()
