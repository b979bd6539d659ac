"""The bounded wait of the resident bricks for one another: a budget of 0 looks, with which no
block waits at all, is reported once as LBM_ETIMEOUT, and the context then steps as a new one
does (needs a GPU)."""
import numpy as np
import pytest

from paper_1507_07294_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_1507_07294_gb300 import lbm
    lbm.load_library()
    return lbm


def _budget(L, s, polls):
    L.lbm_set_tuning(s.ctx, L.LBM_TUNE_TMA_WAIT_POLLS, polls)
    L.lbm_set_tuning(s.ctx, L.LBM_TUNE_BRICKS, 1)
    assert L.lbm_get_tuning(s.ctx, L.LBM_TUNE_BRICKS) == 1


REPORTS = {  # calls that report it; each takes its own steps or none
    "reduce": lambda L, s: s.reduce(),
    "step_reduce": lambda L, s: L.lbm_step_reduce(s.ctx, 3),
    "fields": lambda L, s: s.fields(L.LBM_FIELD_PHI),
}


@pytest.mark.parametrize("report", list(REPORTS))
@pytest.mark.parametrize("tracking", [False, True])
@pytest.mark.parametrize("pattern,storage", [("ab", "fp32"), ("ab", "fp16"), ("aa", "fp32"), ("aa", "bf16")])
def test_a_wait_that_runs_out(L, pattern, storage, tracking, report):
    w = I.perturbed(I.droplet(R=5.0, nx=32, ny=16, nz=24), seed=71, phi_amp=0.02, u_amp=0.01)
    if tracking:
        w.velocity = ("rotation", 0.001)
    with L.Solver(w, pattern=pattern, storage=storage) as a, \
            L.Solver(w, pattern=pattern, storage=storage) as b:
        default = L.lbm_get_tuning(a.ctx, L.LBM_TUNE_TMA_WAIT_POLLS)
        a.step(3)
        b.step(3)
        _budget(L, a, 0)
        a.step(5)  # two calls are queued before either is reported
        a.step(4)
        with pytest.raises(L.LbmError) as e:
            REPORTS[report](L, a)
        assert e.value.status == L.LBM_ETIMEOUT
        L.lbm_reduce(a.ctx, check=False)  # reported once: raises on any status but LBM_EUNSTABLE
        _budget(L, a, default)
        a.set_state(*b.state())
        for n in (1, 4, 2):
            a.step(n)
            b.step(n)
            sa, sb = a.state(), b.state()
            for k in (0, 2) if tracking else (0, 1, 2):  # tracking leaves the flow lattice alone
                assert np.array_equal(sa[k], sb[k])
            if not tracking:
                ra, rb = L.lbm_step_reduce(a.ctx, 2), L.lbm_step_reduce(b.ctx, 2)
                assert ra[0] == rb[0] and np.array_equal(ra[1], rb[1])
