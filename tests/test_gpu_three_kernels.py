"""The passes of the three-kernel step against one another on small grids, where lbm_step takes
the resident bricks unless a parameter of that step, or LBM_TUNE_BRICKS 0, asks for it (needs a
GPU)."""
import numpy as np
import pytest

from paper_1507_07294_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_1507_07294_gb300 import lbm
    lbm.load_library()
    return lbm


def _workload(shape, walls=False, **kw):
    nx, ny, nz = shape
    w = I.perturbed(I.droplet(R=max(1.0, min(shape) / 4), nx=nx, ny=ny, nz=nz), seed=sum(shape),
                    phi_amp=0.02, u_amp=0.01, p_amp=1e-3)
    w.walls_z = walls
    if walls:
        w.g = (0.0, 0.0, -1e-5)
    for k, v in kw.items():
        setattr(w, k, v)
    return w


PARAMETERS = ["PREFETCH_COLLIDE", "PREFETCH_PHI", "PREFETCH_COLLIDE_SUMS", "MU_TMA", "GRAPHS",
              "TMA_WAIT_POLLS", "ROWS", "FUSED", "FUSED_SEGMENT", "FUSED_PREFETCH", "CELL_PAIRS",
              "STENCIL_STAGE"]


@pytest.mark.parametrize("name", PARAMETERS)
def test_setting_a_parameter_of_the_passes_asks_for_them(L, name):
    """Even to the value that it has."""
    param = getattr(L, "LBM_TUNE_" + name)
    with L.Solver(_workload((64, 16, 24))) as s:
        assert L.lbm_get_tuning(s.ctx, L.LBM_TUNE_BRICKS) == 1
        L.lbm_set_tuning(s.ctx, param, L.lbm_get_tuning(s.ctx, param))
        assert L.lbm_get_tuning(s.ctx, L.LBM_TUNE_BRICKS) == 0
        L.lbm_set_tuning(s.ctx, L.LBM_TUNE_BRICKS, 1)
        assert L.lbm_get_tuning(s.ctx, L.LBM_TUNE_BRICKS) == 1


def test_autotune_leaves_the_bricks_as_they_were(L):
    from paper_1507_07294_gb300 import tune
    with L.Solver(_workload((32, 32, 32))) as s:
        for on in (1, 0):
            L.lbm_set_tuning(s.ctx, L.LBM_TUNE_BRICKS, on)
            tune.autotune(s.ctx, steps=1, warm=1)
            assert L.lbm_get_tuning(s.ctx, L.LBM_TUNE_BRICKS) == on


def _compare(L, w, storage, param, off):
    """Default passes against the same step with one of them set to `off`."""
    with L.Solver(w, storage=storage) as a, L.Solver(w, storage=storage) as b:
        L.lbm_set_tuning(b.ctx, param, off)
        for s in (a, b):
            L.lbm_set_tuning(s.ctx, L.LBM_TUNE_BRICKS, 0)
            assert L.lbm_get_tuning(s.ctx, L.LBM_TUNE_BRICKS) == 0
        assert L.lbm_get_tuning(a.ctx, param) != off == L.lbm_get_tuning(b.ctx, param)
        for n in (1, 2, 5):
            for s in (a, b):
                s.step(n)
            for x, y in zip(a.state()[:3], b.state()[:3]):
                assert np.array_equal(x, y)
        for n in (1, 3):
            ra, rb = L.lbm_step_reduce(a.ctx, n), L.lbm_step_reduce(b.ctx, n)
            assert ra[0] == rb[0] and np.array_equal(ra[1], rb[1])
        for x, y in zip(a.state()[:3], b.state()[:3]):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("name", ["PREFETCH_COLLIDE", "PREFETCH_PHI", "PREFETCH_COLLIDE_SUMS",
                                  "MU_TMA", "GRAPHS", "ROWS", "CELL_PAIRS"])
def test_a_pass_and_its_alternative_give_the_same_bits(L, name, storage, walls):
    _compare(L, _workload((64, 16, 24), walls), storage, getattr(L, "LBM_TUNE_" + name), 0)


@pytest.mark.parametrize("variant", [{"srt_flow": True}, {"stencil": "d3q7"},
                                     {"srt_flow": True, "stencil": "d3q7"}])
@pytest.mark.parametrize("name", ["CELL_PAIRS", "GRAPHS"])
def test_the_variants(L, name, variant):
    _compare(L, _workload((64, 16, 24), True, **variant), "fp32", getattr(L, "LBM_TUNE_" + name), 0)


@pytest.mark.parametrize("grid", [(32, 1, 1, False), (32, 3, 5, True), (64, 1, 2, True),
                                  (64, 8, 9, False), (96, 5, 7, True)])
@pytest.mark.parametrize("storage", ["fp32", "bf16"])
def test_row_addressing(L, grid, storage):
    _compare(L, _workload(grid[:3], grid[3]), storage, L.LBM_TUNE_ROWS, 0)


def test_single_pass_against_three(L):
    w = _workload((64, 16, 24), True)
    with L.Solver(w) as a, L.Solver(w) as b:
        L.lbm_set_tuning(a.ctx, L.LBM_TUNE_FUSED, 1)
        L.lbm_set_tuning(b.ctx, L.LBM_TUNE_BRICKS, 0)
        assert L.lbm_get_tuning(a.ctx, L.LBM_TUNE_FUSED) == 1
        assert L.lbm_get_tuning(b.ctx, L.LBM_TUNE_BRICKS) == 0
        for n in (1, 4):
            a.step(n)
            b.step(n)
            for x, y in zip(a.state()[:3], b.state()[:3]):
                assert np.array_equal(x, y)
