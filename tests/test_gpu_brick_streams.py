"""Which contexts on several streams step in resident bricks: those whose launches fit the device
together (needs a GPU)."""
import numpy as np
import pytest

from paper_1507_07294_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_1507_07294_gb300 import lbm
    lbm.load_library()
    return lbm


def _bricks(L, *solvers):
    return [L.lbm_get_tuning(s.ctx, L.LBM_TUNE_BRICKS) for s in solvers]


def _streams(n):
    import torch
    return [torch.cuda.Stream() for _ in range(n)]


def test_full_launches_of_two_streams(L):
    """48^3 takes 432 of 456 places.  Steps on either side of the change give the same bits."""
    w = I.perturbed(I.droplet(n=48, R=12.0), seed=3, u_amp=0.01)
    q, r = _streams(2)
    with L.Solver(w, stream=q.cuda_stream) as a, L.Solver(w, stream=q.cuda_stream) as ref:
        assert _bricks(L, a, ref) == [1, 1]  # one stream: in turn
        a.step(3)
        with L.Solver(w, stream=r.cuda_stream) as b:
            assert _bricks(L, a, b) == [0, 0]
            a.step(4)
            b.step(2)
            L.lbm_set_tuning(b.ctx, L.LBM_TUNE_BRICKS, 0)  # its short launches overlap
            assert _bricks(L, a, b) == [1, 0]
            L.lbm_set_tuning(b.ctx, L.LBM_TUNE_BRICKS, 1)
            assert _bricks(L, a, b) == [0, 0]
        assert _bricks(L, a) == [1]
        a.step(2)
        L.lbm_set_tuning(ref.ctx, L.LBM_TUNE_BRICKS, 0)
        ref.step(9)
        for x, y in zip(a.state()[:3], ref.state()[:3]):
            assert np.array_equal(x, y)


def test_launches_that_fit_together(L):
    """32^3 takes 128 of 456 places: three streams do, four do not; 16^3 takes 64."""
    w = I.droplet(n=32, R=8.0)
    solvers = [L.Solver(w, stream=q.cuda_stream) for q in _streams(3)]
    try:
        assert _bricks(L, *solvers) == [1, 1, 1]
        solvers.append(L.Solver(w, stream=_streams(1)[0].cuda_stream))
        small = [L.Solver(I.droplet(n=16, R=4.0), stream=q.cuda_stream) for q in _streams(6)]
        solvers += small
        assert _bricks(L, *solvers) == [0] * 4 + [1] * 6
    finally:
        for s in solvers:
            s.close()


def test_threads_step_at_once(L):
    """Contexts made, stepped and closed by several threads: the states of one at a time."""
    import threading
    w = I.perturbed(I.droplet(n=32, R=8.0), seed=4, u_amp=0.01)
    with L.Solver(w) as s:
        s.step(30)
        want = s.state()[:3]
    got, errors = [None] * 6, []

    def work(k, stream):
        try:
            for _ in range(3):
                with L.Solver(w, stream=stream.cuda_stream) as s:
                    for n in (1, 9, 20):
                        s.step(n)
                    got[k] = s.state()[:3]
        except Exception as e:  # reported by the main thread
            errors.append(e)

    streams = _streams(6)
    threads = [threading.Thread(target=work, args=(k, q)) for k, q in enumerate(streams)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for g in got:
        for x, y in zip(g, want):
            assert np.array_equal(x, y)
