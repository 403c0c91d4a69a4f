"""The choices the library makes by size, alignment and call pattern give the
results of the general path: graph-launched steps, the geometry's thread and
warp paths on both sides of their line, 16-cell flag preparation with
obstacles, and field read-back into buffers of either alignment."""
import ctypes as C

import numpy as np
import pytest

from paper_1409_5645_gb300 import cases, fslbm, slabs
from tests.gpu_util import run_parity

pytestmark = pytest.mark.gpu


def _splash(precision, **kw):
    c = cases.dam_break(nx=72, ny=24, nz=32, col_x=24, col_z=22, tau=0.6, g=2e-4, rule=1, **kw)
    return c, lambda **o: fslbm.Lattice.from_case(c, precision=precision, **o)


def _same(a, b):
    ga, gb = a.get(63), b.get(63)
    return all(np.array_equal(ga[k], gb[k]) for k in ga)


@pytest.mark.parametrize("precision,loads", [("f64", "plain"), ("f32", "pairs"), ("f16", "plain")])
def test_steps_by_graph_equal_single_steps(precision, loads):
    """19 steps in one call (two graphs of eight steps and three of one) equal
    19 calls, timed steps (kernel by kernel) and steps after a change of the
    schedule or of the owned region."""
    c, make = _splash(precision, bulk_loads=loads)
    a, b, t = make(), make(), make()
    a.step(19)
    for _ in range(19):
        b.step(1)
    t.timing(True)
    t.step(19)
    assert _same(a, b) and _same(a, t) and a.time == 19
    assert a.counters() == b.counters() == t.counters()
    # parameters that the captured steps hold: t, kernel by kernel, takes the new ones at once
    a.set_overlap(False)
    for g in (a, b, t):
        g.set_owned((0, 0, 0), (36, 24, 32))
        g.step(9)
    assert _same(a, b) and _same(a, t)
    assert a.step_mass() == pytest.approx(t.step_mass(), rel=1e-12)
    assert b.step_mass() == pytest.approx(t.step_mass(), rel=1e-12)


def test_steps_on_a_captured_stream():
    import torch
    s = torch.cuda.Stream()
    c, make = _splash("f32", bulk_loads="pairs")
    a, b = make(stream=s.cuda_stream), make()
    a.step(10)
    a.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        a.step(2)
    with torch.cuda.stream(s):
        g.replay()
        g.replay()
    s.synchronize()
    b.step(14)
    assert _same(a, b)


@pytest.mark.parametrize("dims,col,periodic", [((40, 30, 24), (20, 16), (0, 0, 0)),      # few cells: a warp each
                                               ((160, 64, 40), (60, 24), (0, 0, 0)),     # interior cells above the line
                                               ((512, 7, 40), (420, 30), (0, 0, 0)),     # edge cells above it
                                               ((512, 7, 40), (420, 30), (0, 1, 0))])    # ... with a periodic axis
def test_geometry_paths_match_the_oracle(dims, col, periodic):
    c = cases.dam_break(nx=dims[0], ny=dims[1], nz=dims[2], col_x=col[0], col_z=col[1], tau=0.6, g=2e-4, rule=1,
                        phi_noise=0.3, periodic=periodic)
    c["phi"] = np.where(c["flags"] == cases.INTERFACE, np.clip(c["phi"], 0.05, 0.999), c["phi"])
    run_parity(c, 2)


@pytest.mark.parametrize("nx,periodic", [(16, (0, 0, 0)), (48, (0, 0, 0)), (48, (1, 1, 0)), (44, (0, 1, 0))])
def test_flag_preparation_with_obstacles(nx, periodic):
    """Obstacles of WALL cells inside the liquid, across group borders and at
    the faces, in rows of whole 16-cell groups and in others."""
    c = cases.dam_break(nx=nx, ny=10, nz=14, col_x=nx // 2, col_z=9, tau=0.7, g=2e-4, rule=1, periodic=periodic)
    f = c["flags"].reshape(14, 10, nx)
    phi = c["phi"].reshape(14, 10, nx)
    for z, y, x in ((2, 3, 0), (2, 5, nx // 4), (3, 5, nx // 4 + 1), (4, 9, 5), (0, 4, 3), (5, 6, nx - 1), (1, 7, 15 % nx)):
        f[z, y, x] = cases.WALL
        phi[z, y, x] = 0.0
    run_parity(c, 12, check_mass=False)


def test_bad_states_are_still_refused():
    c = cases.dam_break(nx=48, ny=10, nz=14, col_x=20, col_z=9, tau=0.7, g=2e-4, rule=1)
    for at, kind in ((20 + 48 * (4 + 10 * 4), cases.LIQUID), (3 + 48 * (4 + 10 * 4), 3), (17 + 48 * (5 + 10 * 3), 0)):
        flags = c["flags"].copy()
        flags[at] = kind  # liquid beside gas; two kinds at once; no kind
        g = fslbm.Lattice(c["dims"], c["params"])
        with pytest.raises(fslbm.FslbmError) as e:
            g.init_equilibrium(flags, c["rho"], c["u"], c["phi"])
        assert e.value.code == -4


@pytest.mark.parametrize("dims", [(20, 9, 14), (21, 9, 13)])
def test_fields_into_buffers_of_either_alignment(dims):
    import torch
    c = cases.dam_break(nx=dims[0], ny=dims[1], nz=dims[2], col_x=8, col_z=9, tau=0.7, g=2e-4, rule=1)
    g = fslbm.Lattice.from_case(c, precision="f32")
    g.step(5)
    ref = g.get(63)
    N = g.N
    sizes = {"flags": N, "f": 19 * N, "m": N, "phi": N, "rho": N, "u": 3 * N}
    for off in (0, 1):
        buf = {k: torch.full((n + 4,), 7, dtype=torch.uint8 if k == "flags" else torch.float64, device="cuda")
               for k, n in sizes.items()}
        ptr = (C.c_void_p * 6)(*[t[off:].data_ptr() for t in buf.values()])
        assert g.L.fslbm_get_fields(g.h, 63, ptr, fslbm.DEVICE) == 0
        for k, n in sizes.items():
            got = buf[k].cpu().numpy()
            assert np.array_equal(got[off:off + n], ref[k].reshape(-1)), (k, off)
            assert (got[:off] == 7).all() and (got[off + n:] == 7).all(), (k, off)


@pytest.mark.parametrize("precision", ["f64", "f32", "f16"])
@pytest.mark.parametrize("rule,kw", [(1, {}), (0, {}), (1, dict(tau=1.7, magic=0.25)), (1, dict(linear_eq=1)),
                                     (1, dict(sigma=1e-3)), (0, dict(wall_u=(1e-3, 0.0, 0.0)))])
def test_interface_cells_by_warp_and_by_thread(precision, rule, kw):
    """A lattice with more interface cells than the warp path takes, beside
    itself as two slabs that have fewer: the same bits after 20 steps with
    conversions."""
    c = cases.dam_break(nx=48, ny=40, nz=40, col_x=20, col_z=20, g=4e-4, rule=rule, phi_noise=0.3, **{"tau": 0.6, **kw})
    c["phi"] = np.where(c["flags"] == cases.INTERFACE, np.clip(c["phi"], 0.05, 0.999), c["phi"])
    assert int((c["flags"] == cases.INTERFACE).sum()) > 1216 > 28 * 40
    whole = fslbm.Lattice.from_case(c, precision=precision)
    parts = slabs.LocalSlabs(c, parts=2, axis=1, precision=precision)
    whole.step(20)
    for _ in range(20):
        parts.step(1)
    a, b = whole.get(fslbm.FIELD_FLAGS | fslbm.FIELD_F | fslbm.FIELD_MASS), parts.owned_fields(
        fslbm.FIELD_FLAGS | fslbm.FIELD_F | fslbm.FIELD_MASS)
    assert whole.counters()[4] > 0
    for k in a:
        assert np.array_equal(a[k].reshape(-1), np.asarray(b[k]).reshape(-1)), k


@pytest.mark.parametrize("precision", ["f32", "f16"])
@pytest.mark.parametrize("depth,more", [(80, False), (10, True)])
def test_pair_kernel_grids_beside_the_interface_kernels(precision, depth, more):
    """Fewer and more interface cells than segments of 32 cells (the pair
    kernel keeps fewer blocks where there are more), beside every kernel in
    order on the full grid."""
    c = cases.dam_break(nx=512, ny=6, nz=96, col_x=500, col_z=depth, tau=0.6, g=2e-4, rule=1)
    liquid = (c["flags"] == cases.LIQUID).reshape(-1, 32).any(1).sum()
    assert ((c["flags"] == cases.INTERFACE).sum() > liquid) == more
    a, b = (fslbm.Lattice.from_case(c, precision=precision, bulk_loads="pairs") for _ in range(2))
    b.set_overlap(False)
    for g in (a, b):
        g.step(30)
    assert _same(a, b) and a.counters()[4] > 0
    assert a.step_mass() == pytest.approx(b.step_mass(), rel=1e-12)
