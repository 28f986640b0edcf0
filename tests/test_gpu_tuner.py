"""The tuner times the inverses on blocks laid out as the level's own: packed where the plane assembly packs
them, whole where a rotating frame's source or the tensor-core assembly leaves whole ones."""
import pytest

from workloads import ogrid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("params,packed", [(dict(), True), (dict(omega=(0.0, 0.0, 0.1)), False), (dict(block_kernels=1), False)])
def test_stand_ins_are_packed_where_the_blocks_are(params, packed):
    import paper_1807_01151_gb300 as emg
    s = emg.Solver(ogrid(12, 6), p_max=2, prec=1, **params)
    notes = [n for n in s.tuning.split(";") if "gj B=" in n]
    s.close()
    assert len(notes) == 2
    for n in notes:
        assert ("packed split" in n) == packed and "split" in n, n
