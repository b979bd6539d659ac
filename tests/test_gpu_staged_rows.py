"""The staged stream-collide (k_collide2t) on blocks at the edges of what it copies: rows at the
periodic y faces, the whole of y in one block, rows of several planes in one block, a last block
that is not full -- against the same step with one cell per thread (needs a GPU)."""
import numpy as np
import pytest

from paper_1507_07294_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_1507_07294_gb300 import lbm
    lbm.load_library()
    return lbm


@pytest.mark.parametrize("pattern", ["ab", "aa"])
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("shape", [(64, 1, 9), (64, 2, 7), (64, 3, 5), (64, 4, 4), (64, 5, 5),
                                   (64, 8, 1), (128, 1, 5), (128, 2, 4), (128, 3, 5), (128, 6, 2),
                                   (256, 1, 3), (256, 2, 2), (256, 5, 3)])
def test_staged_equals_one_cell_per_thread(L, shape, walls, pattern):
    nx, ny, nz = shape
    w = I.perturbed(I.droplet(R=3.0, nx=nx, ny=ny, nz=nz), seed=nx + ny + nz, phi_amp=0.05,
                    u_amp=0.01, p_amp=1e-4)
    w.walls_z = walls
    with L.Solver(w, pattern=pattern) as a, L.Solver(w, pattern=pattern) as b:
        L.lbm_set_tuning(a.ctx, L.LBM_TUNE_STENCIL_STAGE, 1)
        assert L.lbm_get_tuning(a.ctx, L.LBM_TUNE_STENCIL_STAGE) == 1
        L.lbm_set_tuning(b.ctx, L.LBM_TUNE_CELL_PAIRS, 0)
        for n in (1, 4):
            a.step(n)
            b.step(n)
            for x, y in zip(a.state()[:3], b.state()[:3]):
                assert (np.asarray(x).view(np.uint32) == np.asarray(y).view(np.uint32)).all()
