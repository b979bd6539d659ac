"""Bricks of which two share an SM and a third is kept out (needs a GPU): the same bits as the
three-kernel step, or for tracking as the in-place pattern's three passes."""
import numpy as np
import pytest

from paper_1507_07294_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_1507_07294_gb300 import lbm
    lbm.load_library()
    return lbm


@pytest.mark.parametrize("shape,tracking", [((97, 105, 57), False), ((128, 110, 43), False),
                                            ((79, 113, 63), False), ((96, 123, 101), True)])
def test_same_bits(L, shape, tracking):
    w = I.droplet(R=10.0, nx=shape[0], ny=shape[1], nz=shape[2])
    w = I.perturbed(w, seed=5, phi_amp=0.02, u_amp=0.01)
    w.walls_z = True
    if tracking:
        w.velocity = ("rotation", 1e-4)
    with L.Solver(w) as a, L.Solver(w, pattern="aa" if tracking else "ab") as b:
        L.lbm_set_tuning(b.ctx, L.LBM_TUNE_BRICKS, 0)
        assert L.lbm_get_tuning(a.ctx, L.LBM_TUNE_BRICKS) == 1
        for n in (1, 4):
            a.step(n)
            b.step(n)
            sa, sb = a.state(), b.state()
            for k in (0, 2) if tracking else (0, 1, 2):
                assert np.array_equal(sa[k].view(np.uint32), sb[k].view(np.uint32))


def test_single_tracking_steps_between_launches_of_many(L):
    """Beyond 350,000 cells a single step is one pass over the box, several are bricks."""
    w = I.perturbed(I.droplet(R=10.0, nx=75, ny=72, nz=70), seed=6, phi_amp=0.02)
    w.velocity = ("deformation", 0.01, 40.0)
    with L.Solver(w) as a, L.Solver(w, pattern="aa") as b:
        L.lbm_set_tuning(b.ctx, L.LBM_TUNE_BRICKS, 0)
        assert L.lbm_get_tuning(a.ctx, L.LBM_TUNE_BRICKS) == 1
        for n in (1, 4, 1, 1, 3):
            a.step(n)
            b.step(n)
            sa, sb = a.state(), b.state()
            for k in (0, 2):
                assert np.array_equal(sa[k].view(np.uint32), sb[k].view(np.uint32))
