"""The staged stream-collide (k_collide2t) in its model variants and with the step sums, on blocks
inside a plane, blocks that span several planes and a last block that is not full, against the
same step with one cell per thread (needs a GPU)."""
import numpy as np
import pytest

from paper_1507_07294_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SHAPES = [(64, 10, 3), (64, 3, 5), (64, 12, 24), (128, 3, 5), (128, 10, 12), (256, 5, 3)]
VARIANTS = {"mrt": {}, "srt": {"srt_flow": True}, "d3q7": {"stencil": "d3q7"},
            "both": {"srt_flow": True, "stencil": "d3q7"}}


@pytest.fixture(scope="module")
def L():
    from paper_1507_07294_gb300 import lbm
    lbm.load_library()
    return lbm


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("variant", list(VARIANTS))
@pytest.mark.parametrize("storage,pattern", [("fp32", "ab"), ("fp32", "aa"), ("fp16", "ab")])
def test_staged_equals_one_cell_per_thread(L, storage, pattern, variant, walls, shape):
    nx, ny, nz = shape
    w = I.perturbed(I.droplet(R=3.0, nx=nx, ny=ny, nz=nz), seed=nx + ny + nz, phi_amp=0.05,
                    u_amp=0.01, p_amp=1e-4)
    w.walls_z = walls
    for k, v in VARIANTS[variant].items():
        setattr(w, k, v)
    with L.Solver(w, pattern=pattern, storage=storage) as a, \
            L.Solver(w, pattern=pattern, storage=storage) as b:
        L.lbm_set_tuning(a.ctx, L.LBM_TUNE_STENCIL_STAGE, 1)
        L.lbm_set_tuning(b.ctx, L.LBM_TUNE_CELL_PAIRS, 0)
        for s in (a, b):
            assert L.lbm_get_tuning(s.ctx, L.LBM_TUNE_BRICKS) == 0
            assert L.lbm_get_tuning(s.ctx, L.LBM_TUNE_STENCIL_STAGE) == (s is a)
        for n in (1, 4):
            for s in (a, b):
                s.step(n)
            for x, y in zip(a.state()[:3], b.state()[:3]):
                assert np.array_equal(x.view(np.uint32), y.view(np.uint32))
        for n in (1, 2):
            ra, rb = L.lbm_step_reduce(a.ctx, n), L.lbm_step_reduce(b.ctx, n)
            assert ra[0] == rb[0] and np.array_equal(ra[1], rb[1])
        for x, y in zip(a.state()[:3], b.state()[:3]):
            assert np.array_equal(x.view(np.uint32), y.view(np.uint32))
