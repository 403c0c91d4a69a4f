"""The stability guard at any u_max: a uniform flow two parts in a thousand
above it is refused, one as far below steps (FP64; the fixed-point collision's
unit of |u|^2, 2^-60, would not tell them apart near 1e-8)."""
import numpy as np
import pytest

from paper_1409_5645_gb300 import cases, fslbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps", [1, 6])
@pytest.mark.parametrize("u_max", [1e-9, 3e-8, 1e-5, 1e-2, 0.4])
def test_guard_resolves_its_bound(u_max, steps):
    dims = (16, 8, 8)
    params = cases.default_params(tau=0.8, periodic=(1, 1, 1))
    flags, zero = np.full(1024, cases.LIQUID, np.uint8), np.zeros(1024)
    for factor in (0.998, 1.002):
        lat = fslbm.Lattice(dims, dict(params, u_max=u_max))
        u = np.zeros((1024, 3))
        u[:, 0] = u_max * factor
        lat.init_equilibrium(flags, np.ones(1024), u, zero)
        if factor < 1:
            lat.step(steps)
            lat.sync()
        else:
            with pytest.raises(fslbm.FslbmError) as e:
                lat.step(steps)
                lat.sync()
            assert e.value.code == -5 and "velocity" in str(e.value)
