"""The resident kernel (many steps per launch, state on chip; the default of small lattices) gives
the bits of one step per launch: fields, phasors and forces, at sizes where strips, segments and
thread blocks are ragged, for every form, polarization and source."""
import numpy as np
import pytest

from paper_2509_22308_gb300 import lbm_em as L

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2509_22308_gb300 import build
    build.build()


def _solver(nx, ny, prec, pol, kind, spl, stream=None):
    """Many materials (a graded band, conductors on it and at the edges), so that no warp's sites
    are all alike, next to rows of pure vacuum."""
    x, y = np.meshgrid(np.arange(nx), np.arange(ny))
    eps = np.where((y > ny // 3) & (y < 2 * ny // 3), 1.0 + ((x * 7 + y * 3) % 40) * 0.1, 1.0)
    pec = ((x % 17 == 5) & (y % 13 == 7)) | ((x == nx - 1) & (y == ny - 1)) | ((x == 0) & (y == ny // 2))
    return L.Solver(nx, ny, prec, eps_map=eps, pec_mask=pec, source=L.make_source(24, 30, kind), stream=stream,
                    steps_per_launch=spl, polarization=pol)


def _same(a, b):
    for u, v in zip(a.fields(), b.fields()):
        assert np.array_equal(u, v)


SHAPES = [(4, 4), (5, 61), (64, 48), (65, 33), (67, 45), (31, 70), (127, 129), (128, 152), (300, 17), (259, 301), (512, 512)]


@pytest.mark.parametrize("kind", [L.SRC_HARD, L.SRC_OPEN])
@pytest.mark.parametrize("prec,pol", [("f64", "tm"), ("f64", "te"), ("f32", "tm"), ("f32", "te"), ("f32x2", "tm"),
                                      ("f32x2", "te")])
@pytest.mark.parametrize("shape", SHAPES)
def test_resident_steps_are_bit_identical(shape, prec, pol, kind):
    nx, ny = shape
    with _solver(nx, ny, prec, pol, kind, "auto") as a, _solver(nx, ny, prec, pol, kind, "one") as b:
        for n in (41, 2, 3, 290):  # resident, plain, resident, two resident launches
            a.step(n)
            b.step(n)
            _same(a, b)
        if min(nx, ny) >= 30:
            c = L.make_contour(min(nx, ny) / 2 - 3.0, 4.0)
            Fa, Fb = a.force_torque(c), b.force_torque(c)
            assert np.array_equal(Fa, Fb)
            a.accumulate(170)
            b.accumulate(170)
            assert np.array_equal(a.phasors()[1], b.phasors()[1])
        a.sync()
        assert a.t == b.t


@pytest.mark.parametrize("prec,shape,own", [("f64", (150, 139), True), ("f32", (150, 139), True), ("f32x2", (150, 139), True),
                                            ("f64", (150, 139), False), ("f32", (341, 350), False), ("f32", (341, 350), True)])
def test_resident_reset_checkpoint_and_streams(prec, shape, own):
    """A reset run repeats its bits, a checkpoint resumes them, and handles whose launches are in
    flight at once do not disturb each other: on the library's streams (where the later ones take plain
    launches or, large FP32 lattices, all take resident ones) and on the caller's."""
    import torch
    nx, ny = shape
    with _solver(nx, ny, prec, "tm", L.SRC_HARD, "one") as ref:
        ref.step(400)
        want = ref.fields()
    streams = [None if own else torch.cuda.Stream() for _ in range(3)]
    solvers = [_solver(nx, ny, prec, "tm", L.SRC_HARD, "auto", s) for s in streams]
    for _ in range(2):
        for s in solvers:
            s.reset()
        for _ in range(4):
            for s in solvers:
                s.step(50)
        saved = solvers[0].save_state()
        for _ in range(4):
            for s in solvers:
                s.step(50)
        for s in solvers:
            s.sync()
            for u, v in zip(s.fields(), want):
                assert np.array_equal(u, v)
    solvers[1].load_state(saved)
    solvers[1].step(200)
    for u, v in zip(solvers[1].fields(), want):
        assert np.array_equal(u, v)
    for s in solvers:
        s.close()


def test_resident_handles_of_several_threads():
    """Threads that create, step and destroy handles at the same time get the bits of one thread."""
    import threading
    with _solver(120, 90, "f64", "tm", L.SRC_HARD, "one") as ref:
        ref.step(300)
        want = ref.fields()
    bad = []

    def work():
        for _ in range(4):
            with _solver(120, 90, "f64", "tm", L.SRC_HARD, "auto") as s:
                for n in (100, 150, 50):
                    s.step(n)
                if not all(np.array_equal(u, v) for u, v in zip(s.fields(), want)):
                    bad.append(1)

    threads = [threading.Thread(target=work) for _ in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_resident_captured_stream_takes_plain_launches():
    """A caller that captures the handle's stream gets plain launches, as before."""
    import torch
    st = torch.cuda.Stream()
    nx, ny = 341, 350
    with _solver(nx, ny, "f32", "tm", L.SRC_HARD, "auto", st) as a, _solver(nx, ny, "f32", "tm", L.SRC_HARD, "one") as b:
        a.step(20)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            a.step(10)
        g.replay()
        torch.cuda.synchronize()
        b.step(30)
        _same(a, b)
