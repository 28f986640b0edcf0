"""The residual's projections with one and with four threads per mode on either side of the element counts
where the choice changes, against the oracle.  The bound is derived in test_gpu_residual_fixed."""
import numpy as np
import pytest

from oracle.dg import DG
from tests.helpers import perturbed_state
from tests.test_gpu_residual_fixed import _largest_terms, _solver
from workloads import cubed_sphere_shell, ogrid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,size,p", [(2, (151, 105), 1), (2, (157, 103), 1), (2, (79, 56), 2), (2, (79, 57), 2),
                                        (3, (4, 8), 3), (3, (4, 9), 3), (3, (3, 8), 4), (3, (3, 9), 4)])
def test_residual_on_either_side_of_the_split(dim, size, p):
    desc = ogrid(*size) if dim == 2 else cubed_sphere_shell(*size)
    dg = DG(desc, p)
    u = perturbed_state(dg, seed=51 + p)
    s = _solver(desc, p)
    R = s.residual(p, u)
    again = s.residual(p, u)   # the kernels of consecutive calls overlap at their ends
    s.close()
    np.testing.assert_array_equal(R, again)
    assert np.abs(R - dg.residual(p, u)).max() <= 32 * 2.0 ** -52 * _largest_terms(dg, p, u)
