"""Ratios of specific heats other than 7/5: the far field's power is pow(x, 1 / (gamma - 1)) in the place of
x^2 sqrt(x), in the residual and in the FP64 and float32 face Jacobians.  The bounds are those of the other
residual and block tests (test_gpu_residual_fixed; float32 blocks: B u32 of the block's norm, times the
face Jacobians' few hundred operations)."""
import numpy as np
import pytest

from oracle.dg import DG
from tests.helpers import perturbed_state
from tests.test_gpu_residual_fixed import _largest_terms
from workloads import cubed_sphere_shell, ogrid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gamma", [1.3, 5.0 / 3.0])
@pytest.mark.parametrize("dim,size,p", [(2, (9, 4), 0), (2, (9, 4), 2), (3, (1, 2), 1)])
def test_residual_and_blocks(dim, size, p, gamma):
    import paper_1807_01151_gb300 as emg
    desc = ogrid(*size) if dim == 2 else cubed_sphere_shell(*size)
    dg = DG(desc, p, gamma=gamma)
    u = perturbed_state(dg, seed=61 + p)
    s = emg.Solver(desc, p_max=p, gamma=gamma)
    R, D = s.residual(p, u), s.jacobian_diag(p, u)
    s.close()
    Do = dg.diag_blocks(p, u)
    if p > 0:
        assert np.abs(R - dg.residual(p, u)).max() <= 32 * 2.0 ** -52 * _largest_terms(dg, p, u)
    else:
        assert np.abs(R - dg.residual(p, u)).max() <= 1e-12 * np.abs(dg.residual(p, u)).max()
    assert np.abs(D - Do).max() <= 1e-11 * np.abs(Do).max()
    if p > 0:
        s = emg.Solver(desc, p_max=p, gamma=gamma, prec=1)
        P = s.block_operator(p, u, cfl=1e12)   # P = I / dtau - D
        s.close()
        B = D.shape[-1]
        assert np.abs(P + Do).max() <= 300 * B * 2.0 ** -24 * np.abs(Do).max()
