"""Results that the host waits for, with and without one of the 64 page-locked slots (needs a
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


def _results(L, s):
    import torch
    page = {"phi": torch.empty(s.ctx.n, dtype=torch.float64, pin_memory=True).numpy()}
    out = [L.lbm_step_reduce(s.ctx, 1), L.lbm_step_reduce(s.ctx, 3), s.reduce()]
    fields = [L.lbm_read_fields(s.ctx, L.LBM_FIELD_PHI, out=page)["phi"].copy(),
              s.fields(L.LBM_FIELD_PHI)["phi"]]
    return out, fields


def test_more_contexts_than_slots(L):
    """The same sums and fields from every context, those beyond the 64th among them, and from
    contexts made after slots came back."""
    w = I.perturbed(I.droplet(n=8, R=3.0), seed=9, u_amp=0.01)
    solvers = [L.Solver(w) for _ in range(70)]
    try:
        want = _results(L, solvers[0])
        for s in solvers[1:]:
            _same(_results(L, s), want)
        for s in solvers[:5]:
            s.close()
        solvers[:5] = [L.Solver(w) for _ in range(5)]
        for s in solvers[:5]:
            _same(_results(L, s), want)
    finally:
        for s in solvers:
            s.close()


def _same(got, want):
    for (m, j), (wm, wj) in zip(got[0], want[0]):
        assert m == wm and np.array_equal(j, wj)
    for f, wf in zip(got[1], want[1]):
        assert np.array_equal(f, wf)


def test_a_timeout_is_reported_without_a_slot(L):
    w = I.perturbed(I.droplet(n=16, R=5.0, nx=64, ny=16, nz=24), seed=51, u_amp=0.01)
    small = I.droplet(n=4, R=1.0)
    others = [L.Solver(small) for _ in range(66)]
    try:
        with L.Solver(w) as s:
            L.lbm_set_tuning(s.ctx, L.LBM_TUNE_TMA_WAIT_POLLS, 0)
            for report in (lambda: s.reduce(), lambda: L.lbm_step_reduce(s.ctx, 1),
                           lambda: s.fields(L.LBM_FIELD_PHI)):
                s.step(1)
                with pytest.raises(L.LbmError) as e:
                    report()
                assert e.value.status == L.LBM_ETIMEOUT
                L.lbm_reduce(s.ctx, check=False)  # reported once
    finally:
        for s in others:
            s.close()
