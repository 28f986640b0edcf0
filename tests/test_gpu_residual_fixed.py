"""The residual's and the FP64 blocks' fixed-point contractions (and the blocks' factorisation) (traces, volume quadrature, projections) against the
oracle: element counts that leave the last block short, both splits of the projection (few
elements: four threads per mode), every order, a spanwise momentum in 2-D, and non-finite input.

Tolerance: each factor is cut at 2^-56 of its group's largest, a sum of K <= 120 terms leaves out
less than K 2^-58 of the largest product, and results are rounded at 2^-53; the point fluxes add a
few float64 roundings.  So every entry is within 32 * 2^-52 of M, the largest sum of absolute terms
|W d_k psi_i| |F| over an element's points plus |psi_i| w |F| over its face points."""
import numpy as np
import pytest

from oracle import euler
from oracle.dg import DG
from tests.helpers import perturbed_state
from workloads import cubed_sphere_shell, ogrid

pytestmark = pytest.mark.gpu


def _solver(desc, p):
    import paper_1807_01151_gb300 as emg
    return emg.Solver(desc, p_max=p)


def _largest_terms(dg, p, u):
    L = dg.levels[p]
    F = np.abs(euler.flux(np.einsum('eai,eqi->eqa', u, L.psi), dg.gamma)[..., :dg.dim, :])
    vol = np.einsum('eqik,eqka->eai', np.abs(L.wgrad), F).max()
    face = (np.abs(L.int_psiL) * L.int_amag[..., None]).sum(1).max() * F.max()
    return vol + 2 * dg.dim * face


CASES = [(2, (5, 3), p) for p in (1, 2, 3, 4)] + [(2, (47, 43), p) for p in (1, 2, 3, 4)] + \
        [(3, (1, 3), p) for p in (1, 2, 3, 4)] + [(3, (7, 7), p) for p in (1, 2)]


@pytest.mark.parametrize("dim,size,p", CASES)
def test_residual_matches_oracle(dim, size, p):
    desc = ogrid(*size) if dim == 2 else cubed_sphere_shell(*size)
    dg = DG(desc, p)
    u = perturbed_state(dg, seed=11 + p)
    s = _solver(desc, p)
    for spanwise in ([False, True] if dim == 2 else [True]):
        if dim == 2 and spanwise:   # every third element carries a spanwise momentum
            u[::3, 3, :] = 0.05 * u[::3, 1, :]
        R = s.residual(p, u)
        err = np.abs(R - dg.residual(p, u)).max()
        assert err <= 32 * 2.0 ** -52 * _largest_terms(dg, p, u)
    s.close()


@pytest.mark.parametrize("size", [(12, 5), (47, 43)])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_coefficient_stays_with_its_neighbours(size, bad):
    desc = ogrid(*size)
    dg = DG(desc, 2)
    u = perturbed_state(dg, seed=3)
    s = _solver(desc, 2)
    clean = s.residual(2, u)
    e = dg.E // 2
    u[e, 1, 2] = bad
    R = s.residual(2, u)
    s.close()
    touched = np.zeros(dg.E, dtype=bool)
    touched[[e] + list(dg.mesh.neighbours[e])] = True
    assert not np.isfinite(R[touched]).all(axis=(1, 2)).any()
    assert np.array_equal(R[~touched], clean[~touched])


@pytest.mark.parametrize("dim,size,p", [(2, (7, 3), 0), (2, (7, 3), 1), (2, (7, 3), 2), (2, (5, 3), 3), (2, (5, 2), 4),
                                        (3, (1, 2), 1), (3, (1, 2), 2), (3, (1, 1), 3)])
def test_diagonal_blocks_match_oracle(dim, size, p):
    """Blocks (face Jacobians and assembly) with and without a spanwise momentum in 2-D; the bound is
    that of the other FP64 block tests."""
    desc = ogrid(*size) if dim == 2 else cubed_sphere_shell(*size)
    dg = DG(desc, p)
    u = perturbed_state(dg, seed=21 + p)
    s = _solver(desc, p)
    for spanwise in ([False, True] if dim == 2 else [True]):
        if dim == 2 and spanwise:
            u[::3, 3, :] = 0.05 * u[::3, 1, :]
        D = s.jacobian_diag(p, u)
        Do = dg.diag_blocks(p, u)
        assert np.abs(D - Do).max() <= 1e-11 * np.abs(Do).max()
        for e in range(dg.E):   # element by element too: their scales differ by the mesh's stretching
            assert np.abs(D[e] - Do[e]).max() <= 1e-11 * np.abs(Do[e]).max()
    s.close()


@pytest.mark.parametrize("size,p", [((7, 3), 1), ((7, 3), 2), ((5, 3), 3), ((5, 2), 4)])
@pytest.mark.parametrize("state,forcing", [(False, False), (True, False), (False, True)])
def test_fp64_prk_step_with_and_without_spanwise_momentum(size, p, state, forcing):
    """The FP64 factorisation splits blocks whose spanwise momentum is uncoupled: plane flow (split,
    spanwise part of the residual 0), plane flow with a spanwise forcing (split, both systems solved)
    and a state with a spanwise momentum (whole blocks).  The bound is that of the FP64 PRK tests."""
    from oracle import emg as oemg
    desc = ogrid(*size)
    dg = DG(desc, p)
    u = perturbed_state(dg, seed=31 + p)
    tau = np.zeros_like(u)
    if state:
        u[::3, 3, :] = 0.05 * u[::3, 1, :]
    if forcing:
        tau[:, 3, :] = 1e-3 * u[:, 0, :]
    s = _solver(desc, p)
    out = s.prk_step(p, u, tau=tau, cfl=5.0)
    s.close()
    D = dg.diag_blocks(p, u)
    P = np.eye(D.shape[-1])[None] / oemg.dtau(dg, p, u, 5.0)[:, None, None] - D
    ref = oemg.prk_step(lambda w: dg.residual(p, w) + tau, P, u)
    assert np.abs(out - ref).max() <= 1e-11 * np.abs(ref).max()
    if not (state or forcing):
        assert not out[:, 3].any()
