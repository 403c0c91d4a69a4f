"""dJ/dnu of films whose terms cancel to 1e-8 of themselves, against the values
of the general reverse collision (each population's term by itself), to 1e-9:
the FP64 reverse collision's roundings are the general form's where it
matters.  (The noise field of 1e-8 makes the remainder; seeds at which the
-3/2 u.u parts summed over the links moved it by 5e-9 to 1.4e-8.)"""
import pytest

from paper_1409_5645_gb300 import cases, fslbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,seed,J,dnu", [((5, 3, 57), 32, 0.02004999944206247, 1.6296650624084045e-10),
                                             ((5, 3, 57), 63, 0.020049999424110235, -9.932847385727788e-10),
                                             ((8, 4, 64), 88, 0.020050000647110634, 1.7417529359287276e-10),
                                             ((8, 4, 64), 15, 0.020049999563938388, -3.156141085686446e-10)])
def test_cancelling_viscosity_gradient(dims, seed, J, dnu):
    c = cases.film(nx=dims[0], ny=dims[1], nz=dims[2], h=round(0.625 * dims[2]), gx=1e-4, noise_amp=1e-8, seed=seed)
    g = fslbm.Lattice.from_case(c, keep_f0=1)
    assert g.adjoint_forward(200, 50) == pytest.approx(J, rel=1e-13)
    assert g.adjoint_backward()[0] == pytest.approx(dnu, rel=1e-9)
