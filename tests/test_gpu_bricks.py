"""The resident-brick steps of small grids (LBM_TUNE_BRICKS) against the three-kernel step:
the same bits for every way a grid is cut -- bricks of one cell, uneven bricks, rows that are
no tiles, axes shorter than a stencil -- and the sums of the last step (needs a GPU)."""
import numpy as np
import pytest

from paper_1507_07294_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_1507_07294_gb300 import lbm
    lbm.load_library()
    return lbm


def _bits(states):
    return [np.asarray(a).view(np.uint32) for a in states[:3]]


def _pair(L, w, storage="fp32", pattern="ab"):
    a, b = (L.Solver(w, storage=storage, pattern=pattern) for _ in range(2))
    L.lbm_set_tuning(b.ctx, L.LBM_TUNE_BRICKS, 0)
    assert L.lbm_get_tuning(a.ctx, L.LBM_TUNE_BRICKS) == 1
    assert L.lbm_get_tuning(b.ctx, L.LBM_TUNE_BRICKS) == 0
    return a, b


def _workload(shape, walls, **kw):
    nx, ny, nz = shape
    w = I.perturbed(I.droplet(R=max(1.0, min(shape) / 4), nx=nx, ny=ny, nz=nz), seed=sum(shape),
                    phi_amp=0.02, u_amp=0.01, p_amp=1e-4)
    w.walls_z = walls
    w.g = (0.0, 0.0, -1e-5)
    for k, v in kw.items():
        setattr(w, k, v)
    return w


@pytest.mark.parametrize("pattern", ["ab", "aa"])
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("shape", [(32, 32, 32), (37, 41, 45), (64, 16, 24), (5, 5, 5), (1, 1, 1),
                                   (3, 4, 400), (256, 8, 3), (1, 7, 2), (33, 1, 70), (64, 48, 56)])
def test_same_bits_as_the_three_kernel_step(L, shape, walls, storage, pattern):
    if pattern == "aa" and np.prod(shape) > 36000:
        pytest.skip("in place the line lies lower")
    a, b = _pair(L, _workload(shape, walls), storage, pattern)
    with a, b:
        for n in (1, 2, 5):
            a.step(n)
            b.step(n)
            sa, sb = a.state(), b.state()
            assert sa[3] == sb[3]
            for x, y in zip(_bits(sa), _bits(sb)):
                assert (x == y).all()
        for n in (1, 3):
            ra, rb = L.lbm_step_reduce(a.ctx, n), L.lbm_step_reduce(b.ctx, n)
            assert ra[0] == rb[0] and (ra[1] == rb[1]).all()


@pytest.mark.parametrize("kw", [{"srt_flow": True}, {"stencil": "d3q7"},
                                {"srt_flow": True, "stencil": "d3q7"}, {"buoyancy": True}])
@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("pattern", ["ab", "aa"])
def test_variants(L, kw, storage, pattern):
    a, b = _pair(L, _workload((40, 24, 30), True, **kw), storage, pattern)
    with a, b:
        a.step(6)
        b.step(6)
        for x, y in zip(_bits(a.state()), _bits(b.state())):
            assert (x == y).all()


@pytest.mark.parametrize("n,kind", [(1, "deformation"), (6, "zalesak"), (32, "zalesak"),
                                    (33, "deformation"), (48, "deformation"), (70, "zalesak")])
@pytest.mark.parametrize("storage", ["fp32", "bf16"])
@pytest.mark.parametrize("pattern", ["ab", "aa"])
def test_tracking(L, n, kind, storage, pattern):
    """More steps than one launch has time factors for; a single left-over step among them."""
    if pattern == "aa" and n ** 3 > 270000:
        pytest.skip("in place the line lies lower")
    w = I.deformation(n=n, period=100.0) if kind == "deformation" else I.zalesak(n=n)
    a, b = _pair(L, w, storage, pattern)
    with a, b:
        for k in (1, 65, 130):
            a.step(k)
            b.step(k)
        sa, sb = a.state(), b.state()
        assert (_bits(sa)[0] == _bits(sb)[0]).all() and (_bits(sa)[2] == _bits(sb)[2]).all()


def test_long_runs_and_where_it_applies(L):
    """More steps than a launch takes; grids beyond the line, profiling and a changed parameter of the three-kernel step go through that step."""
    a, b = _pair(L, _workload((16, 16, 16), False))
    with a, b:
        a.step(1025)
        b.step(1025)
        for x, y in zip(_bits(a.state()), _bits(b.state())):
            assert (x == y).all()
        L.lbm_profile(a.ctx, True)
        assert L.lbm_get_tuning(a.ctx, L.LBM_TUNE_BRICKS) == 0
        L.lbm_profile(a.ctx, False)
        L.lbm_set_tuning(a.ctx, L.LBM_TUNE_GRAPHS, 0)
        assert L.lbm_get_tuning(a.ctx, L.LBM_TUNE_BRICKS) == 0
        with pytest.raises(L.LbmError):
            L.lbm_set_tuning(a.ctx, L.LBM_TUNE_BRICKS, 2)
    with L.Solver(I.droplet(n=8, R=2.0, nx=87, ny=86, nz=86)) as s:  # 643,452 cells
        assert L.lbm_get_tuning(s.ctx, L.LBM_TUNE_BRICKS) == 0


def test_a_captured_step_replays(L):
    """Under capture the three-kernel step is recorded, so that a replay does its work."""
    import torch
    w = _workload((32, 32, 32), False)
    st = torch.cuda.Stream()
    with L.Solver(w, stream=st.cuda_stream) as a, L.Solver(w) as b:
        a.step(2)
        b.step(3)
        st.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            a.step(1)
        with torch.cuda.stream(st):
            graph.replay()
        for x, y in zip(_bits(a.state()), _bits(b.state())):
            assert (x == y).all()
