"""Rows of 3 cells of 2^20 x 1 (x 2^10) in a uniform flow along x between symmetry planes, whose mirrored
states are the inside ones to the last bit: equal states have no Roe dissipation, so the fluxes of mass,
x momentum and energy through the long faces are 0, and a cell's residual is 0 as the difference of
sums of the short faces' size.  The fixed-point contractions keep the small gradients along the long side.

Bound of an entry, for any form that sums its own terms in 53 bits: the sum of its own absolute terms times
(2 N^2 + 64) 2^-53, N^2 twice for the set-up's Gram-Schmidt basis (N modes, two roundings in each of N
projections), 64 for the sums and point fluxes."""
import numpy as np
import pytest

from oracle import euler
from oracle.dg import DG
from workloads import BC_FARFIELD, BC_INTERIOR, BC_SYMMETRY, MeshDesc

pytestmark = pytest.mark.gpu


def cell_row(dim, sides):
    """Three cells along x, from the origin."""
    corner = [(0, 0), (1, 0), (1, 1), (0, 1)]
    corner = corner if dim == 2 else [c + (k,) for k in (0, 1) for c in corner]
    nodes = [(i,) + c for i in range(4) for c in np.ndindex(*(2,) * (dim - 1))]
    en = [[nodes.index((i + c[0],) + c[1:]) for c in corner] for i in range(3)]
    fb = np.full((3, 2 * dim), BC_SYMMETRY, dtype=np.int32)
    fb[:, :2] = BC_INTERIOR
    fb[0, 0] = fb[2, 1] = BC_FARFIELD
    return MeshDesc(dim, np.array(nodes, dtype=float).T * np.array(sides)[:, None], np.array(en, dtype=np.int64), fb,
                    name="row")


def own_terms(dg, p, u):
    """Sum of the absolute terms of every entry of the residual."""
    L, m = dg.levels[p], dg.mesh
    F = np.abs(euler.flux(np.einsum("eai,eqi->eqa", u, L.psi), dg.gamma)[..., :dg.dim, :])
    S = np.einsum("eqik,eqka->eai", np.abs(L.wgrad), F)
    UL = np.einsum("fai,fqi->fqa", u[m.int_L], L.int_psiL)
    UR = np.einsum("fai,fqi->fqa", u[m.int_R], L.int_psiR)
    Fh = np.abs(L.int_amag[..., None] * euler.roe(UL, UR, L.int_n, dg.gamma))
    np.add.at(S, m.int_L, np.einsum("fqi,fqa->fai", np.abs(L.int_psiL), Fh))
    np.add.at(S, m.int_R, np.einsum("fqi,fqa->fai", np.abs(L.int_psiR), Fh))
    return S


def entries(dim, p):
    """Residual of the middle cell (mass, x momentum, energy), the sums of its terms, the bound's factor."""
    import paper_1807_01151_gb300 as emg
    desc = cell_row(dim, (2.0 ** 20, 1.0, 2.0 ** 10)[:dim])
    dg = DG(desc, p)
    u = dg.freestream_state(p)
    s = emg.Solver(desc, p_max=p)
    R = s.residual(p, u)
    s.close()
    S = own_terms(dg, p, u)[1, [0, 1, 4]]
    assert S.min() > 0
    return np.abs(R[1, [0, 1, 4]]), S, (2 * dg.N(p) ** 2 + 64) * 2.0 ** -53


@pytest.mark.parametrize("dim,p", [(2, 1), (2, 2), (2, 4), (3, 1), (3, 3)])
def test_no_dissipation_between_equal_states(dim, p):
    err, S, c = entries(dim, p)
    assert (err[:, 0] <= c * S[:, 0]).all(), (err / S)[:, 0].max() / c


@pytest.mark.parametrize("dim,p", [(2, 1), (2, 2), (2, 3), (2, 4), (3, 1), (3, 2), (3, 3), (3, 4)])
def test_residual_entries_of_stretched_cells(dim, p):
    err, S, c = entries(dim, p)
    assert (err <= c * S).all(), (err / S).max() / c


def own_block_terms(dg, p, u, e):
    """Sum of the absolute terms of every entry [a][b][i][j] of element e's block, its interior faces only."""
    L, m = dg.levels[p], dg.mesh

    def slope(f, x):   # df_a/dx_b by complex steps
        d = [f(x + 1e-30j * np.eye(5)[b]).imag / 1e-30 for b in range(5)]
        return np.abs(np.stack(d, -1))

    U = np.einsum("ai,qi->qa", u[e], L.psi[e])
    S = 0.0
    for k in range(dg.dim):
        A = slope(lambda x: euler.flux(x, dg.gamma)[:, k], U)
        S = S + np.einsum("qi,qab,qj->abij", np.abs(L.wgrad[e, :, :, k]), A, np.abs(L.psi[e]))
    for f in range(len(m.int_L)):
        UL, UR = L.int_psiL[f] @ u[m.int_L[f]].T, L.int_psiR[f] @ u[m.int_R[f]].T
        flux = lambda l, r: L.int_amag[f][:, None] * euler.roe(l, r, L.int_n[f], dg.gamma)
        for side, psi, J in ((m.int_L, L.int_psiL, slope(lambda x: flux(x, UR + 0j), UL)),
                             (m.int_R, L.int_psiR, slope(lambda x: flux(UL + 0j, x), UR))):
            if side[f] == e:
                S = S + np.einsum("ti,tab,tj->abij", np.abs(psi[f]), J, np.abs(psi[f]))
    return S


@pytest.mark.parametrize("dim,p", [(2, 1), (2, 2), (2, 3), (2, 4), (3, 1), (3, 2), (3, 3)])
def test_block_entries_of_stretched_cells(dim, p):
    """The FP64 blocks: mass, x momentum and energy by density, x momentum and energy, which the long faces
    (exactly: the mirrored state's part cancels the inside one's) add nothing to."""
    import paper_1807_01151_gb300 as emg
    desc = cell_row(dim, (2.0 ** 20, 1.0, 2.0 ** 10)[:dim])
    dg = DG(desc, p)
    u = dg.freestream_state(p)
    s = emg.Solver(desc, p_max=p)
    D = s.jacobian_diag(p, u)[1]
    s.close()
    n = dg.N(p)
    err = np.abs(D - dg.diag_blocks(p, u)[1]).reshape(5, n, 5, n).transpose(0, 2, 1, 3)
    S = own_block_terms(dg, p, u, 1)
    c = (2 * n * n + 64) * 2.0 ** -53
    for a, b in ((0, 1), (1, 0), (1, 1), (4, 0), (4, 1)):
        ok = S[a, b] > 1e-12 * S[a, b].max()   # not where all the terms are the set-up's rounding
        assert ok.any() and (err[a, b] <= c * S[a, b])[ok].all(), (a, b, (err[a, b][ok] / S[a, b][ok]).max() / c)
