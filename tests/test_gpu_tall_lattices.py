"""Lattices of more rows than one step kernel's grid can have blocks for (65535 along y)."""
import numpy as np
import pytest

from paper_2509_22308_gb300 import lbm_em as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny", [262140, 262141, 262147])
def test_tall_double_float_lattice_steps(ny):
    """Around the last height that the packed double-float kernel's blocks of 4 rows reach.  The plane wave in
    vacuum has the same bits in every row, so the rows are those of a low lattice."""
    def fields(rows):
        with L.Solver(4, rows, "f32x2", eps_map=np.ones((rows, 4)), source=L.make_source(8, 4),
                      steps_per_launch="one") as s:
            s.step(2)
            s.step(9)
            s.sync()
            return s.fields()
    for tall, low in zip(fields(ny), fields(16)):
        assert np.array_equal(low, np.broadcast_to(low[0], low.shape))
        assert np.array_equal(tall, np.broadcast_to(low[0], tall.shape))
    assert np.any(low)
