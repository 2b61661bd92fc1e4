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


def test_remainders_of_two_and_three_steps():
    """Calls of 2, 3, 6 and 7 steps from even and odd times, with and without Fourier sums: the bits of one step per
    launch.  A call of two steps takes no longer than with two steps per launch throughout."""
    import torch
    with _solver(720, 730) as a, _solver(720, 730, "one") as b:
        assert a.steps_per_launch() == 4
        c = L.make_contour(100.0, 50.0, cx=110.0)
        for s in (a, b):
            for n in (2, 3, 6, 7, 1, 2, 3, 7):
                s.step(n)
            s.set_contour(c)
            for n in (2, 3, 6, 7, 1, 2, 3, 7):
                s.accumulate(n)
        assert a.t == b.t and np.any(a.phasors()[1])
        assert np.array_equal(a.phasors()[1], b.phasors()[1])
        for u, v in zip(a.fields(), b.fields()):
            assert np.array_equal(u, v)

    def us(s):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = 1e9
        for _ in range(20):
            e0.record(st)
            for _ in range(50):
                s.step(2)
            e1.record(st)
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        return best

    st = torch.cuda.Stream()
    kw = dict(janus=L.make_janus(100.0, 0.4, 2.0, 3.0), source=L.make_source(24), stream=st)
    with L.Solver(900, 900, "f32", **kw) as a, L.Solver(900, 900, "f32", steps_per_launch="two", **kw) as b:
        assert a.steps_per_launch() == 4
        # (single steps: 1.24 times)
        assert us(a) < 1.12 * us(b)
