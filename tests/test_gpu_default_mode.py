"""The steps per launch that FP32 lattices between 2^19 and 2^20 sites take by default, and their bits."""
import numpy as np
import pytest

from paper_2509_22308_gb300 import lbm_em as L

pytestmark = pytest.mark.gpu


def _solver(nx, ny, spl="auto"):
    return L.Solver(nx, ny, "f32", janus=L.make_janus(min(nx, ny) / 6.0, 0.4, 2.0, 3.0), source=L.make_source(24),
                    steps_per_launch=spl)


# strips of 56 columns against tiles of 64: twice as many, 1.5, 1.25 and 1.0 times; padded rows that leave L2; flat
# and tall lattices; lattices from 2^20 sites on
@pytest.mark.parametrize("nx,ny,mode", [(60, 9000, 2), (64, 16383, 2), (64, 16384, 4), (57, 12000, 2), (57, 18200, 4), (128, 4140, 2),
                                        (113, 5000, 2), (256, 2070, 2), (256, 3000, 4), (100, 5300, 4), (112, 4700, 4),
                                        (400, 1325, 4), (724, 725, 4), (900, 900, 4), (723, 725, 2), (131072, 4, 4), (4, 131072, 4)])
def test_half_empty_strips_keep_two_steps_per_launch(nx, ny, mode):
    with _solver(nx, ny) as a, _solver(nx, ny, "one") as b:
        assert a.steps_per_launch() == mode
        a.step(39)
        b.step(39)
        for u, v in zip(a.fields(), b.fields()):
            assert np.array_equal(u, v)
