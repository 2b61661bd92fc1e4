"""The double-float step on packed pairs of rows against the scalar one.

A launch without Fourier sums takes the packed kernel, one with them the scalar one; the operations are
the same, so the fields after the same steps have the same bits."""
import numpy as np
import pytest

from paper_2509_22308_gb300 import lbm_em as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pol", ["tm", "te"])
@pytest.mark.parametrize("nx,ny,kind", [(12, 12, L.SRC_HARD), (33, 9, L.SRC_HARD), (64, 47, L.SRC_OPEN),
                                        (97, 130, L.SRC_HARD), (31, 64, L.SRC_NONE)])
def test_packed_rows_have_the_scalar_bits(nx, ny, kind, pol):
    T, n = 16, 60
    rng = np.random.default_rng(nx + ny)
    eps = rng.uniform(1.0, 6.0, 4)[rng.integers(0, 4, (ny, nx))]
    pec = (rng.random((ny, nx)) < 0.05).astype(np.uint8)
    out = []
    for accumulate in (False, True):
        with L.Solver(nx, ny, "f32x2", eps_map=eps, pec_mask=pec, source=L.make_source(T, kind=kind),
                      polarization=pol, steps_per_launch="one") as s:
            if accumulate:
                a = min(nx, ny) / 8.0
                s.set_contour(L.make_contour(1.2 * a, a))
                s.accumulate(n)
            else:
                s.step(n)
            out.append(s.fields())
    for u, v in zip(*out):
        assert np.array_equal(u, v) and (kind == L.SRC_NONE or np.any(u))
