"""Convergence exits of the FP32 batch: four-step launches between the period boundaries against
one-step launches throughout.

The one-step kernel takes the steps that sample the energy, so both paths sample the same sites' same
values; only the order in which thread blocks add their sums differs, which decides an exit only if
the change of energy equals the tolerance to 1e-15.  Run lengths are therefore equal and forces
have the same bits."""
import numpy as np
import pytest

from paper_2509_22308_gb300 import lbm_em as L

pytestmark = pytest.mark.gpu


def _inst(nx, ny, period, periods, **kw):
    a = min(nx, ny) / 6.0
    return dict(dict(nx=nx, ny=ny, a=a, phi0=0.4, eps1=2.0, eps2=3.0, pec2=False, period=period, periods=periods,
                     R=min(nx, ny) / 3.5, ramp=period), **kw)


@pytest.mark.parametrize("pol", ["tm", "te"])
@pytest.mark.parametrize("periods_of", [(24, 24, 24, 24), (25, 25, 25, 25), (30, 45, 30, 61), (27, 27, 90, 27)])
def test_four_step_launches_between_period_boundaries(periods_of, pol):
    """One period of 4 k, 4 k + 1 steps, and several at once (runs that end between the others'
    boundaries, at their maximum and early); a second run of the same batch starts afresh."""
    T = periods_of
    insts = [_inst(64, 48, T[0], 40), _inst(57, 61, T[1], 40, eps2=9.0), _inst(128, 56, T[2], 3),
             _inst(200, 73, T[3], 30, pec2=True, phi0=1.9)]
    out = []
    for kw in ({}, {"steps_per_launch": 1}):
        b = L.Batch(insts, "f32", conv_tol=2e-3, min_periods=4, polarization=pol, **kw)
        try:
            assert b.steps_per_launch() == (1 if kw else 4)
            for _ in range(2):
                b.run()
                F, st = b.results()
                assert (st == L.OK).all()
                out.append((F, b.steps()))
        finally:
            b.close()
    full = np.array([i["period"] * i["periods"] for i in insts])
    assert (out[0][1] < full).any() and out[0][1][2] == full[2]
    for F, steps in out[1:]:
        assert np.array_equal(F, out[0][0]) and np.array_equal(steps, out[0][1])


def test_many_different_periods_keep_one_step_launches():
    """Where period boundaries leave few gaps of four steps, the batch stays on the one-step kernel."""
    insts = [_inst(40, 36, 8 + k, 12) for k in range(12)]
    b, c = L.Batch(insts, "f32", conv_tol=1e-2), L.Batch(insts, "f32", conv_tol=1e-2, steps_per_launch=1)
    try:
        assert b.steps_per_launch() == 1
        b.run(), c.run()
        assert np.array_equal(b.steps(), c.steps()) and np.array_equal(b.results()[0], c.results()[0])
    finally:
        b.close(), c.close()


@pytest.mark.parametrize("n", [1, 33, 60])
def test_shorter_segments_as_runs_end(n):
    """Units of 16 rows from the start (one instance), and longer ones that shorten as runs of 2 to 10
    periods end: forces equal the one-step kernel's bits."""
    insts = [_inst(150 + 7 * (k % 9), 260 - 11 * (k % 7), 20 + k % 3, 2 + k % 9) for k in range(n)]
    F = []
    for spl in (4, 1):
        b = L.Batch(insts, "f32", steps_per_launch=spl)
        try:
            b.run()
            F.append(b.results()[0])
        finally:
            b.close()
    assert np.array_equal(F[0], F[1])
