"""Interface cells by a thread each (long lists) and by a warp each (up to 1216
cells): the same bits for every closure of the default instances.  A lattice
that is periodic along y, beside itself laid k times along y, has the same
cells; only the long one's list is above the line.  (Calls of four steps: the
step's kernels.)"""
import numpy as np
import pytest

from paper_1409_5645_gb300 import cases, fslbm

pytestmark = pytest.mark.gpu


def _along_y(c, k):
    nx, ny, nz = c["dims"]

    def lay(a, comps):
        if a is None:
            return None
        if comps == 3:
            return np.tile(a.reshape(nz, ny, nx, 3), (1, k, 1, 1)).reshape(-1, 3)
        if comps == 19:
            return np.tile(a.reshape(19, nz, ny, nx), (1, 1, k, 1)).reshape(-1)
        return np.tile(a.reshape(nz, ny, nx), (1, k, 1)).reshape(-1)

    return cases.Case(dims=(nx, ny * k, nz), params=c["params"], flags=lay(c["flags"], 1), rho=lay(c["rho"], 1),
                      u=lay(c["u"], 3), phi=lay(c["phi"], 1), noise=lay(c["noise"], 19),
                      wall_delta=lay(c["wall_delta"], 19))


def _film(cli=False, **kw):
    """A film with a rough surface (open and closed columns, cells near their
    thresholds), walls below, and with cli link fractions there and at an obstacle."""
    args = dict(nx=12, ny=10, nz=20, h=11.5, tau=0.6, gx=2e-4, noise_amp=2e-3)
    args.update(kw)
    c = cases.film(**args)
    ifc = c["flags"] == cases.INTERFACE
    c["phi"] = np.where(ifc, np.clip(c["phi"] + cases.uniform(3, c.N, 0.45), 0.02, 0.98), c["phi"])
    if cli:
        flags, phi = c["flags"].reshape(20, 10, 12), c["phi"].reshape(20, 10, 12)
        flags[4:13, 3:5, 5:7] = cases.WALL  # (through the surface: interface cells at the obstacle)
        phi[4:13, 3:5, 5:7] = 0.0
        c["wall_delta"] = 0.5 + cases.uniform(8, 19 * c.N, 0.45)
    return c


CASES = [("inclined_cli_shift", lambda: cases.inclined_film(), 100, ("f64", "f32", "f16")),
         ("inclined_cli_fsk", lambda: cases.inclined_film(rule=0), 100, ("f64", "f32", "f16")),
         ("film_fsl", lambda: _film(), 12, ("f64", "f32", "f16")),
         ("film_fsk", lambda: _film(rule=0), 12, ("f64", "f32", "f16")),
         ("film_cli", lambda: _film(cli=True), 12, ("f64", "f32", "f16")),
         ("film_sigma", lambda: _film(sigma=1e-3), 12, ("f64", "f32", "f16")),
         ("film_gas_density", lambda: _film(rho_G=0.99, sigma=1e-3, rule=0), 12, ("f64", "f32", "f16")),
         ("film_delta_min", lambda: _film(delta_min=0.1), 12, ("f64", "f32", "f16")),
         ("film_linear", lambda: _film(linear_eq=1), 12, ("f32", "f16")),
         ("film_compressible", lambda: _film(compressible=1), 12, ("f32",)),
         ("film_moving_wall", lambda: _film(wall_u=(1e-3, 5e-4, 0.0), h=2.5), 12, ("f64", "f32", "f16")),
         ("film_frozen", lambda: _film(freeze=1), 12, ("f64", "f32", "f16"))]


@pytest.mark.parametrize("precision,make,k",
                         [pytest.param(p, make, k, id=f"{name}-{p}") for name, make, k, ps in CASES for p in ps])
def test_thread_and_warp_cells_give_the_same_bits(precision, make, k):
    c = make()
    nx, ny, nz = c["dims"]
    long_ = _along_y(c, k)
    assert int((c["flags"] == cases.INTERFACE).sum()) * 2 < 1216 < int((long_["flags"] == cases.INTERFACE).sum())
    a = fslbm.Lattice.from_case(c, precision=precision, u_max=0.0)
    b = fslbm.Lattice.from_case(long_, precision=precision, u_max=0.0)
    for _ in range(4):
        for _ in range(3):
            a.step(4)
            b.step(4)
        assert a.counters()[4] <= 1216 < b.counters()[4]
        fa, fb = a.get(63), b.get(63)
        for key, v in fb.items():
            tail = v.shape[1:] if key == "u" else ()
            lead = (19,) if key == "f" else ()
            v = v.reshape(*lead, nz, k, ny, nx, *tail)
            w = fa[key].reshape(*lead, nz, 1, ny, nx, *tail)
            same = (v == w) | ((v != v) & (w != w))
            assert same.all(), f"{key} differs at {np.argwhere(~same)[:4].tolist()}"
    a.sync()
    b.sync()
