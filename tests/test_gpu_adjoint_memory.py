"""The buffers that a differentiation leaves with its handle: used again by the
next one of the same window, given back by a second new state without one, and
the gradients are those of a fresh handle either way."""
import numpy as np
import pytest

from paper_1409_5645_gb300 import cases, fslbm

pytestmark = pytest.mark.gpu


def test_buffers_are_kept_for_one_state_and_given_back():
    import torch
    c = cases.dam_break(nx=96, ny=48, nz=64, col_x=32, col_z=40, tau=0.6, g=2e-4, rule=1)
    g = fslbm.Lattice.from_case(c, precision="f32", keep_f0=1)

    def state():
        g.init_equilibrium(c["flags"], c["rho"], c["u"], c["phi"])

    def free():
        g.sync()
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    def gradient():
        J = g.adjoint_forward(6, 3)
        return J, *g.adjoint_backward()

    # the handle's graphs, and what the driver keeps for kernels once they have run
    for _ in range(20):
        g.step(8)
    other = fslbm.Lattice.from_case(c, precision="f32", keep_f0=1)
    other.adjoint_forward(6, 3)
    other.adjoint_backward()
    other.close()
    state()
    before, mib = free(), 2 ** 20
    first = gradient()
    held = before - free()
    assert held > 100 * mib  # (three adjoint fields alone are 19 * 8 * 3 N bytes)
    state()
    assert before - free() > held - 16 * mib  # one new state: kept
    again = gradient()
    assert before - free() < held + 16 * mib  # and used
    state()
    state()
    assert before - free() < 16 * mib  # a second one: given back
    third = gradient()
    for other in (again, third):
        assert other[0] == first[0]
        # (the reverse sweep adds some adjoints by atomics, in any order)
        assert other[1] == pytest.approx(first[1], rel=1e-11)
        assert np.abs(other[3] - first[3]).max() <= 1e-11 * np.abs(first[3]).max()
