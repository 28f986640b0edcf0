"""The float32 blocks of 2-D levels: blocks whose spanwise momentum is uncoupled are assembled, inverted
and applied as two systems; the others go through lists to the kernels of whole blocks.  Element counts
that leave the assembly's last block short, every order, and plane flow, plane flow with a spanwise
forcing (split blocks, spanwise right-hand side) and a spanwise momentum in some elements (a mixture).

Bounds: the assembly forms sum the same terms in the same order, so their blocks are equal.  Inverse:
Gauss-Jordan with partial pivoting, ||X^ - X|| / ||X|| <= 4 kappa_2(P) B u32 (u32 = 2^-24).  PRK step
(four stages, each within kappa_2 B u32 of the float64 solve with the same blocks): the update within
8 max kappa_2(P) B u32."""
import numpy as np
import pytest

from oracle import emg as oemg
from oracle.dg import DG
from tests.helpers import perturbed_state, rel_err
from workloads import ogrid

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24


@pytest.mark.parametrize("size,p", [((7, 3), 1), ((11, 9), 1), ((7, 3), 2), ((5, 3), 3), ((5, 3), 4)])
@pytest.mark.parametrize("flow", ["plane", "forced", "mixed"])
@pytest.mark.parametrize("prec", [1, 2])
def test_fp32_blocks_with_and_without_spanwise_momentum(size, p, flow, prec):
    import paper_1807_01151_gb300 as emg
    desc = ogrid(*size)
    dg = DG(desc, p)
    u = perturbed_state(dg, seed=41 + p, amp=0.002)
    tau = np.zeros_like(u)
    if flow == "mixed":
        u[::7, 3, :] = 0.05 * u[::7, 1, :]
    if flow == "forced":
        tau[:, 3, :] = 1e-3 * u[:, 0, :]
    cfl = 3.0
    s = emg.Solver(desc, p_max=p, prec=prec)
    P = s.block_operator(p, u, cfl=cfl, which=0).astype(np.float64)
    X = s.block_operator(p, u, cfl=cfl, which=1)
    out = s.prk_step(p, u, tau=tau, cfl=cfl)
    again = s.prk_step(p, u, tau=tau, cfl=cfl)   # the lists' lengths are back at 0
    s.close()
    np.testing.assert_array_equal(out, again)
    if prec == 1:
        s = emg.Solver(desc, p_max=p, prec=1, block_kernels=3)
        np.testing.assert_array_equal(P, s.block_operator(p, u, cfl=cfl, which=0))
        s.close()
    N = P.shape[-1] // 5
    w = np.arange(5 * N) // N == 3
    coupled = (P[:, w][:, :, ~w] != 0).any(axis=(1, 2)) | (P[:, ~w][:, :, w] != 0).any(axis=(1, 2))
    assert coupled.any() == (flow == "mixed") and not coupled.all()
    bound = 4 * np.linalg.cond(P) * 5 * N * U32
    Xo = np.linalg.inv(P)
    err = np.linalg.norm(X - Xo, ord=2, axis=(1, 2)) / np.linalg.norm(Xo, ord=2, axis=(1, 2))
    assert np.all(err <= bound), (err / bound).max()
    ref = oemg.prk_step(lambda v: dg.residual(p, v) + tau, P, u)
    assert rel_err(out - u, ref - u) <= 2 * bound.max()
    if flow == "plane":
        assert not out[:, 3].any()


@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_split_inverse_variants_are_bitwise_the_same(p):
    """Every tuned number of warps gives the same inverses as the untuned choice."""
    import paper_1807_01151_gb300 as emg
    desc = ogrid(9, 5)
    u = perturbed_state(DG(desc, p), seed=5)
    X = []
    for tune in (0, 1):
        s = emg.Solver(desc, p_max=p, prec=1, autotune=tune)
        X.append(s.block_operator(p, u, cfl=20.0, which=1))
        s.close()
    np.testing.assert_array_equal(X[0], X[1])
