"""Which launches a handle's steps take: on-chip ones of many steps where they apply (counted by the library, so
that a comparison with one step per launch cannot pass by comparing plain launches with themselves), plain
ones elsewhere, and the same bits either way at the ends of the on-chip range."""
import numpy as np
import pytest

from paper_2509_22308_gb300 import lbm_em as L

pytestmark = pytest.mark.gpu


def _solver(nx, ny, prec, pol="tm", kind=L.SRC_HARD, spl="auto", stream=None):
    """Many materials in a band (graded, with conductors), vacuum elsewhere."""
    x, y = np.meshgrid(np.arange(nx), np.arange(ny))
    eps = np.where((y > ny // 3) & (y < 2 * ny // 3), 1.0 + ((x * 7 + y * 3) % 40) * 0.1, 1.0)
    pec = ((x % 17 == 5) & (y % 13 == 7)) | ((x == nx - 1) & (y == ny - 1)) | ((x == 0) & (y == ny // 2))
    return L.Solver(nx, ny, prec, eps_map=eps, pec_mask=pec, source=L.make_source(24, 30, kind), stream=stream,
                    steps_per_launch=spl, polarization=pol)


# FP32: seven rows per warp (600^2, ragged, tall), five (wide and 25 high); the largest FP64 segments; double-float
# at its two rows per warp, ragged and tall
ENDS = [("f32", 600, 600), ("f32", 577, 611), ("f32", 300, 1100), ("f32", 6001, 25), ("f64", 540, 540), ("f64", 533, 547),
        ("f32x2", 256, 256), ("f32x2", 341, 337), ("f32x2", 31, 1900)]


@pytest.mark.parametrize("pol,kind", [("tm", L.SRC_HARD), ("te", L.SRC_HARD), ("tm", L.SRC_OPEN), ("te", L.SRC_OPEN)])
@pytest.mark.parametrize("prec,nx,ny", ENDS)
def test_on_chip_launches_at_the_ends_of_their_range(prec, nx, ny, pol, kind):
    with _solver(nx, ny, prec, pol, kind) as a, _solver(nx, ny, prec, pol, kind, "one") as b:
        for s in (a, b):
            s.step(41)
            s.step(270)
        assert a.resident_launches() == 3 and b.resident_launches() == 0
        for u, v in zip(a.fields(), b.fields()):
            assert np.array_equal(u, v) and np.any(u)
        # (where the wave has arrived)
        c = L.make_contour(min(nx, ny) / 2 - 3.0, 4.0, cx=20.0 if nx > 1000 else None)
        for s in (a, b):
            s.set_contour(c)
            s.accumulate(150)
        assert a.resident_launches() == 5
        assert np.array_equal(a.phasors()[1], b.phasors()[1]) and np.any(a.phasors()[1])
        a.sync()
        for u, v in zip(a.fields(), b.fields()):
            assert np.array_equal(u, v)


@pytest.mark.parametrize("prec,nx,ny,own,resident", [
    ("f32", 64, 48, True, True), ("f64", 64, 48, True, True), ("f32x2", 64, 48, True, True), ("f16dev", 64, 48, True, False),
    ("f32", 64, 48, False, False), ("f64", 64, 48, False, False), ("f32", 341, 350, False, True),
    ("f32", 700, 700, True, False), ("f64", 700, 700, True, False), ("f32x2", 512, 512, True, False)])
def test_which_handles_take_on_chip_launches(prec, nx, ny, own, resident):
    import torch
    st = None if own else torch.cuda.Stream()
    with L.Solver(nx, ny, prec, janus=L.make_janus(6.0, 0.4, 2.0), source=L.make_source(24), stream=st) as s:
        s.step(2)
        assert s.resident_launches() == 0
        s.step(3)
        s.sync()
        assert (s.resident_launches() > 0) == resident
    for spl in ("one", "two", "three", "four"):
        if prec == "f32" and nx < 400:
            with L.Solver(nx, ny, prec, janus=L.make_janus(6.0, 0.4, 2.0), source=L.make_source(24), stream=st,
                          steps_per_launch=spl) as s:
                s.step(40)
                s.sync()
                assert s.resident_launches() == 0


def test_a_captured_stream_and_steps_in_flight_elsewhere_take_plain_launches():
    import torch
    st = torch.cuda.Stream()
    with _solver(341, 350, "f32", stream=st) as a:
        a.step(20)
        n = a.resident_launches()
        assert n == 1
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            a.step(10)
        assert a.resident_launches() == n
        g.replay()
        torch.cuda.synchronize()
        a.step(20)
        assert a.resident_launches() == n + 1
    with _solver(150, 139, "f64") as a, _solver(150, 139, "f64") as b:
        b.step(10)
        b.sync()
        a.step(20000)  # some tens of milliseconds
        b.step(50)
        assert a.resident_launches() == 79 and b.resident_launches() == 1
        a.sync()
        b.step(50)
        b.sync()
        assert b.resident_launches() == 2


# the handle that is in flight, the on-chip one beside it, and whether that takes on-chip launches meanwhile
BESIDE = [
    (("f16dev", 512, "auto"), ("f32", 512), False), (("f32", 512, "two"), ("f32", 350), False), (("f32", 512, "two"), ("f32", 128), False),
    (("f64", 600, "auto"), ("f64", 256), False), (("f32x2", 512, "auto"), ("f32x2", 200), False),
    (("f32", 400, "auto"), ("f32", 512), True),     # both on chip and of the size that always is
    (("f32", 2048, "auto"), ("f64", 128), True), (("f32", 800, "auto"), ("f64", 256), True),  # four steps per launch
    (("f64", 1100, "auto"), ("f32", 400), True),    # fills the GPU by itself
    (("f16dev", 256, "auto"), ("f64", 128), True)]  # little in the way of FP64


# (on a caller's stream only FP32 from 330^2 sites on is on chip)
@pytest.mark.parametrize("first,second,resident,streams", [
    (*b, st) for b in BESIDE for st in ("own", "caller's", "one") if st == "own" or (b[1][0] == "f32" and b[1][1] >= 330)])
def test_steps_in_flight_of_other_kinds(first, second, resident, streams):
    import torch
    (prec_a, na, spl), (prec_b, nb) = first, second
    st = {"own": [None, None], "caller's": [torch.cuda.Stream(), torch.cuda.Stream()], "one": [torch.cuda.Stream()] * 2}[streams]
    j, src = L.make_janus(20.0, 0.4, 2.0, 3.0), L.make_source(24)
    with L.Solver(na, na, prec_a, janus=j, source=src, stream=st[0], steps_per_launch=spl) as a, \
            L.Solver(nb, nb, prec_b, janus=j, source=src, stream=st[1]) as b, \
            L.Solver(nb, nb, prec_b, janus=j, source=src, stream=st[1], steps_per_launch="one") as ref:
        b.step(48)
        b.sync()
        n = b.resident_launches()
        assert n == 1
        a.step(20000)  # 25 ms and more
        b.step(48)
        ref.step(96)
        assert b.resident_launches() - n == int(resident or streams == "one")  # (one stream: nothing runs beside it)
        a.sync()
        b.step(48)
        ref.step(48)
        assert b.resident_launches() - n == 1 + int(resident or streams == "one")
        for u, v in zip(b.fields(), ref.fields()):
            assert np.array_equal(u, v)
