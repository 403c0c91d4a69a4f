"""One call of n steps gives the bits of n calls of one step, whichever way the
steps go out: many steps of a small lattice (up to 65 536 cells) in one
launch, graphs of eight steps and of one on a larger one, kernels one by one
(calls of up to four steps never take the many-steps launch)."""
import numpy as np
import pytest

from paper_1409_5645_gb300 import cases, fslbm

pytestmark = pytest.mark.gpu


def _same(a, b, where=""):
    ga, gb = a.get(63), b.get(63)
    for k in ga:
        assert np.array_equal(ga[k], gb[k]), f"{k} differs {where}"
    assert a.counters() == b.counters() and a.time == b.time


def _dam(**kw):
    args = dict(nx=24, ny=10, nz=16, col_x=9, col_z=12, tau=0.6, g=2e-4)
    args.update(kw)
    return cases.dam_break(**args)


def _cli_dam():
    """Wall link fractions on every face and at obstacles, with conversions."""
    c = _dam()
    flags, phi = c["flags"].reshape(16, 10, 24), c["phi"].reshape(16, 10, 24)
    flags[2:4, 3:6, 4:6] = cases.WALL
    phi[2:4, 3:6, 4:6] = 0.0
    c["wall_delta"] = 0.5 + cases.uniform(11, 19 * c.N, 0.45)
    return c


SMALL = [("inclined_cli_shift_frozen", lambda: cases.inclined_film(), ("f64", "f32", "f16")),
         ("plate_moving_wall_frozen", lambda: cases.plate_flow(), ("f64", "f32", "f16")),
         ("wave_sigma", lambda: cases.standing_wave(n=32, depth=16.0, sigma=1e-3, phi_noise=1e-2), ("f64", "f32", "f16")),
         ("droplet_sigma_periodic_frozen", lambda: cases.droplet(n=20, R=5.0), ("f64", "f32", "f16")),
         ("film_fsl", lambda: cases.film(nx=5, ny=6, nz=40, h=25.0, gx=1e-4), ("f64", "f32", "f16")),
         ("film_fsk", lambda: cases.film(nx=5, ny=6, nz=40, h=25.0, gx=1e-4, rule=0), ("f64", "f32", "f16")),
         ("dam_fsk", lambda: _dam(rule=0), ("f64", "f32", "f16")),
         ("dam_weighted_split", lambda: _dam(excess_split=1), ("f64", "f32", "f16")),
         ("dam_moving_wall", lambda: _dam(wall_u=(1e-3, 0.0, 0.0)), ("f64", "f32", "f16")),
         ("dam_cli", _cli_dam, ("f64", "f32", "f16")),
         ("dam_linear", lambda: _dam(linear_eq=1), ("f64", "f32", "f16")),
         ("dam_compressible", lambda: _dam(compressible=1), ("f64", "f32"))]


@pytest.mark.parametrize("precision,make", [pytest.param(p, make, id=f"{name}-{p}") for name, make, ps in SMALL for p in ps])
def test_many_steps_equal_single_steps(precision, make):
    """Odd calls, so that the second one starts from the other buffers."""
    c = make()
    assert c.N <= 65536
    a, b = (fslbm.Lattice.from_case(c, precision=precision) for _ in range(2))
    conversions = 0
    for call in range(3):
        a.step(23)
        for _ in range(23):
            b.step(1)
            conversions += sum(b.counters()[:4])
        _same(a, b, f"after call {call}")
        (ma, la), (mb, lb) = a.total_mass(), b.total_mass()
        assert ma == pytest.approx(mb, rel=1e-14) and la == pytest.approx(lb, rel=1e-12, abs=1e-15)
        assert a.step_mass() == pytest.approx(b.step_mass(), rel=1e-12)
    a.sync()
    if not c["params"]["freeze"] and c["dims"][0] == 24:
        assert conversions > 0


@pytest.mark.parametrize("precision,loads", [("f64", "plain"), ("f32", "pairs"), ("f32", "plain"), ("f16", "pairs")])
def test_eight_step_graphs_follow_the_handles_parameters(precision, loads):
    """Above the many-steps lattices: calls of nineteen, nine and eight steps
    (graphs of eight and of one) against timed steps, which go kernel by kernel:
    from either buffer side, after a change of the schedule, of the owned
    region, and with link fractions given and taken away."""
    c = cases.dam_break(nx=96, ny=32, nz=32, col_x=32, col_z=22, tau=0.6, g=2e-4, rule=1)
    assert c.N > 65536
    a, t = (fslbm.Lattice.from_case(c, precision=precision, bulk_loads=loads) for _ in range(2))
    t.timing(True)

    def both(n):
        for g in (a, t):
            g.step(n)
        _same(a, t, f"after {n} steps")
        assert a.step_mass() == pytest.approx(t.step_mass(), rel=1e-12)

    both(19)  # (now on the second buffers)
    both(9)
    both(8)
    a.set_overlap(False)  # (t keeps the overlap: the same bits)
    both(9)
    for g in (a, t):
        g.set_owned((0, 0, 0), (12, 32, 32))
    both(17)
    whole = a.step_mass()
    for g in (a, t):
        g.set_owned((0, 0, 0), (96, 32, 32))
    both(8)
    assert a.step_mass() != pytest.approx(whole, rel=1e-3)
    wd = 0.5 + cases.uniform(5, 19 * c.N, 0.3)
    for delta in (wd, None):
        for g in (a, t):
            g.init_equilibrium(c["flags"], c["rho"], c["u"], c["phi"], None, delta)
        both(17)


LOADS = [("f32", "async"), ("f32", "pairs"), ("f16", "async"), ("f16", "pairs"), ("f64", "plain")]


@pytest.mark.parametrize("precision,loads", LOADS)
@pytest.mark.parametrize("make", [lambda: _dam(nx=70, ny=12, nz=20, col_x=33, col_z=15, g=3e-4),
                                  lambda: _dam(nx=70, ny=12, nz=20, col_x=33, col_z=15, g=3e-4, rule=0),
                                  lambda: _dam(nx=38, ny=9, nz=11, col_x=12, col_z=7),
                                  lambda: cases.inclined_film(), lambda: cases.plate_flow()],
                         ids=["ragged", "ragged_fsk", "odd", "inclined_film_cli", "plate_flow_moving_wall"])
def test_short_calls_take_the_step_kernels(precision, loads, make):
    """Calls of four steps: the bulk kernel of each kind of loads beside the
    interface kernels, against the plain loads with every kernel in order (after
    set_overlap(False) no call takes the many-steps launch) and against one call
    of all the steps."""
    c = make()
    a = fslbm.Lattice.from_case(c, precision=precision, bulk_loads=loads)
    b, m = (fslbm.Lattice.from_case(c, precision=precision) for _ in range(2))
    assert a.bulk_loads == loads
    b.set_overlap(False)
    for _ in range(5):
        for _ in range(10):
            a.step(4)
        b.step(40)
        m.step(40)
        _same(a, b)
        _same(a, m)


def test_async_loads_on_odd_rows():
    c = _dam(nx=37, ny=9, nz=11, col_x=12, col_z=7)
    for precision in ("f32", "f16"):
        a = fslbm.Lattice.from_case(c, precision=precision, bulk_loads="async")
        b = fslbm.Lattice.from_case(c, precision=precision)
        b.set_overlap(False)
        for _ in range(40):
            a.step(3)
        b.step(120)
        _same(a, b)
