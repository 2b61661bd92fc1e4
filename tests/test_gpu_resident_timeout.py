"""The bounded waits between the thread blocks of an on-chip launch: a block whose messages never come (one that
the test leaves out of the launch) makes the others give up, in about one limit whatever the number of rows
that wait, the library reports LBM_EM_ETIMEOUT and refuses the handle's further steps, and the device stays
usable."""
import time

import numpy as np
import pytest

from paper_2509_22308_gb300 import lbm_em as L

pytestmark = pytest.mark.gpu

LIMIT = 200_000_000  # clock cycles: about 0.1 s


def _solver(prec, nx, ny):
    return L.Solver(nx, ny, prec, janus=L.make_janus(12.0, 0.4, 2.0, 3.0), source=L.make_source(24))


# FP32 tiles of 1, 4 and 7 rows per warp (from 600^2 on a warp can wait for 7 rows of a lost tile's
# columns), and the 8-byte forms, whose warps wait for flags, inboxes and mailboxes
@pytest.mark.parametrize("prec,nx,ny", [("f32", 130, 90), ("f32", 512, 512), ("f32", 600, 600), ("f64", 150, 139),
                                        ("f64", 300, 60), ("f32x2", 150, 139)])
def test_lost_messages_end_the_launch_and_the_handle(prec, nx, ny):
    with _solver(prec, nx, ny) as s:
        s.step(40)
        s.sync()
        s.lose_messages(LIMIT)
        t0 = time.perf_counter()
        s.step(40)
        with pytest.raises(L.LbmEmError) as e:
            s.sync()
        took = time.perf_counter() - t0
        assert e.value.status == L.ETIMEOUT and "message" in str(e.value)
        with pytest.raises(L.LbmEmError) as e:
            s.step(1)
        assert e.value.status == L.ESTATE
        # one limit at a clock between 1 and 2.1 GHz, not one per row
        assert 0.09 < took < 0.35
    with _solver(prec, nx, ny) as a, L.Solver(nx, ny, prec, janus=L.make_janus(12.0, 0.4, 2.0, 3.0),
                                              source=L.make_source(24), steps_per_launch="one") as b:
        a.step(40)
        b.step(40)
        a.sync()
        for u, v in zip(a.fields(), b.fields()):
            assert np.array_equal(u, v)


def test_lost_messages_hook_refuses_other_handles():
    with L.Solver(64, 64, "f32", janus=L.make_janus(9.0, 0.4, 2.0), source=L.make_source(24),
                  steps_per_launch="one") as s:
        for limit, status in ((0, L.EINVAL), (2_000_000_001, L.EINVAL), (1000, L.ESTATE)):
            with pytest.raises(L.LbmEmError) as e:
                s.lose_messages(limit)
            assert e.value.status == status
        s.step(5)
        s.sync()
