"""2-D flow with a spanwise momentum in every element: all blocks go through the lists of whole blocks, with
more entries than the CTAs that share them (so a CTA's shared memory serves several elements), twice.

Bounds: the float32 assembly forms sum the same terms in the same order (equal blocks); Gauss-Jordan with
partial pivoting ||X^ - X|| / ||X|| <= 4 kappa_2(P) B u32; a PRK step's update within twice that of the
float64 one with the same blocks, and within 1e-11 of the state in the FP64 form (as the other tests of
these forms)."""
import numpy as np
import pytest

from oracle import emg as oemg
from oracle.dg import DG
from tests.helpers import perturbed_state, rel_err
from workloads import ogrid

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def flow():
    desc = ogrid(61, 41)   # 2501 elements; the lists' CTAs: 2432 at most
    dg = DG(desc, 1)
    u = perturbed_state(dg, seed=7, amp=0.002)
    u[:, 3, :] = 0.05 * u[:, 1, :]
    return desc, dg, u


@pytest.mark.parametrize("prec", [0, 1])
def test_every_block_listed(flow, prec):
    import paper_1807_01151_gb300 as emg
    desc, dg, u = flow
    cfl = 3.0
    s = emg.Solver(desc, p_max=1, prec=prec)
    P = s.block_operator(1, u, cfl=cfl, which=0).astype(np.float64)
    out = [s.prk_step(1, u, cfl=cfl) for _ in range(2)]
    X = s.block_operator(1, u, cfl=cfl, which=1) if prec else None
    s.close()
    np.testing.assert_array_equal(out[0], out[1])
    ref = oemg.prk_step(lambda v: dg.residual(1, v), P, u)
    if prec == 0:
        assert np.abs(out[0] - ref).max() <= 1e-11 * np.abs(ref).max()
        return
    s = emg.Solver(desc, p_max=1, prec=1, block_kernels=3)
    np.testing.assert_array_equal(P, s.block_operator(1, u, cfl=cfl, which=0))
    s.close()
    bound = 4 * np.linalg.cond(P) * 15 * 2.0 ** -24
    Xo = np.linalg.inv(P)
    assert (np.linalg.norm(X - Xo, ord=2, axis=(1, 2)) <= bound * np.linalg.norm(Xo, ord=2, axis=(1, 2))).all()
    assert rel_err(out[0] - u, ref - u) <= 2 * bound.max()
