"""The division of the Krylov rows over thread blocks: row counts that leave the last block, or its last
warps, without rows, one block, and (m = 40) the form without rows in registers; both forms of the process
against the oracle and bitwise against each other.  The bound is that of the other FP64 EXP1 tests."""
import numpy as np
import pytest

from oracle import emg as oemg
from oracle.dg import DG
from tests.helpers import perturbed_state, rel_err
from workloads import cubed_sphere_shell, ogrid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mk,m", [(lambda: ogrid(5, 3), 30), (lambda: ogrid(13, 5), 30), (lambda: ogrid(29, 9), 30),
                                  (lambda: ogrid(29, 9), 40), (lambda: cubed_sphere_shell(3, 5), 30)])
def test_exp1_step_over_row_counts(mk, m):
    import paper_1807_01151_gb300 as emg
    desc = mk()
    dg = DG(desc, 0)
    u0 = np.ascontiguousarray(perturbed_state(dg, amp=0.05, seed=9)[:, :, :1])
    tau0 = 1e-4 * np.random.default_rng(3).standard_normal(u0.shape)
    dt = oemg.dtau(dg, 0, u0, 100.0) * 2.0
    out = []
    for coop in (1, 0):
        s = emg.Solver(desc, p_max=0, coop_krylov=coop, krylov_m=m)
        out.append(s.exp1_step(u0, dt, tau0))
        s.close()
    np.testing.assert_array_equal(out[0][0], out[1][0])
    assert out[0][1] == out[1][1]
    uo, ko = oemg.exp1_step(dg, u0, tau0, dt, oemg.Options(krylov_m=m))
    assert out[0][1] == ko
    assert rel_err(out[0][0] - u0, uo - u0) < 1e-11
