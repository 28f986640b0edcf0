"""States of negative density and pressure have no Roe average (sqrt(rho_L), sqrt(rho_R)): the residual of
such a state, and its face Jacobians, are NaN, as the oracle's.  U -> -U keeps velocities, enthalpies and
c^2 = gamma p / rho, so only the densities' signs show it; both sides of every face are negative here."""
import numpy as np
import pytest

from oracle.dg import DG
from tests.helpers import perturbed_state
from workloads import cubed_sphere_shell, ogrid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,size,p", [(2, (9, 4), 0), (2, (9, 4), 2), (3, (2, 2), 1)])
def test_negative_densities_on_both_sides_give_nan(dim, size, p):
    import paper_1807_01151_gb300 as emg
    desc = ogrid(*size) if dim == 2 else cubed_sphere_shell(*size)
    dg = DG(desc, p)
    u = perturbed_state(dg, seed=5)
    s = emg.Solver(desc, p_max=p)
    assert np.isfinite(s.residual(p, u)).all()
    R, D = s.residual(p, -u), s.jacobian_diag(p, -u)
    s.close()
    with np.errstate(invalid="ignore"):
        Ro = dg.residual(p, -u)
    mass = np.isnan(Ro[:, 0, 0])
    assert mass.all()
    assert np.isnan(R[:, 0, 0]).all() and np.isnan(D).any(axis=(1, 2)).all()
