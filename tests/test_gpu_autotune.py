"""What the autotuner tries and sets (needs a GPU)."""
import pytest

from paper_1507_07294_gb300 import inputs as I
from paper_1507_07294_gb300 import tune

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_1507_07294_gb300 import lbm
    lbm.load_library()
    return lbm


@pytest.mark.parametrize("nx", [64, 192, 33])  # staged stencils, two cells per thread, one
def test_candidates_reach_a_wave(L, nx):
    """An FP16 run's default is one wave of the two-cell kernel's blocks, which the FP32 run's
    kernels hold at most."""
    w = I.droplet(R=3.0, nx=nx, ny=4, nz=4)
    with L.Solver(w, storage="fp16") as s:
        wave = L.lbm_get_tuning(s.ctx, L.LBM_TUNE_PREFETCH_COLLIDE)
    with L.Solver(w) as s:
        out = tune.autotune(s.ctx, steps=1, warm=1)
    for name in ("prefetch_collide", "prefetch_collide_sums"):
        tried = sorted(int(k) for k in out[name]["ms"])
        assert tried[0] == 0 and tried[-1] >= wave
        # a third and a half of a wave within a tenth of it
        assert all(min(abs(t - f * wave) for t in tried) <= 0.1 * wave for f in (1 / 3, 1 / 2))


@pytest.mark.parametrize("storage,pattern", [("fp32", "ab"), ("fp16", "ab"), ("fp32", "aa")])
def test_tracking_keeps_what_its_steps_do_not_launch(L, storage, pattern):
    """The order-parameter pass of a run that tracks in one pass runs in its read-outs only."""
    w = I.deformation(n=32, period=100.0)
    with L.Solver(w, storage=storage, pattern=pattern) as s:
        phi = L.lbm_get_tuning(s.ctx, L.LBM_TUNE_PREFETCH_PHI)
        out = tune.autotune(s.ctx, steps=1, warm=1)
        one_pass = storage == "fp32" and pattern == "ab"
        assert (out["prefetch_phi"]["ms"] == {}) == one_pass
        if one_pass:
            assert L.lbm_get_tuning(s.ctx, L.LBM_TUNE_PREFETCH_PHI) == phi > 0
        assert L.lbm_get_tuning(s.ctx, L.LBM_TUNE_PREFETCH_PHI) == out["prefetch_phi"]["value"]
