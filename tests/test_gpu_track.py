"""The one-pass tracking step (pattern AB, FP32; bricks off) against the three passes, which the
in-place pattern takes: the same bits at the edges of columns, segments and bricks, on rows that
are tiles and rows that are not (needs a GPU)."""
import numpy as np
import pytest

from paper_1507_07294_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_1507_07294_gb300 import lbm
    lbm.load_library()
    return lbm


@pytest.mark.parametrize("kind", [("deformation", 0.02, 50.0), ("rotation", 0.001), ("uniform", 0.02)])
@pytest.mark.parametrize("walls,stencil", [(False, "d3q15"), (True, "d3q15"), (True, "d3q7")])
@pytest.mark.parametrize("shape", [(32, 8, 32), (32, 1, 1), (64, 7, 33), (96, 17, 65), (32, 9, 31),
                                   (1, 1, 1), (5, 7, 9), (33, 8, 8), (31, 17, 70), (100, 30, 20)])
def test_one_pass_equals_three(L, shape, walls, stencil, kind):
    nx, ny, nz = shape
    w = I.perturbed(I.droplet(R=max(1.0, min(shape) / 3), D=2.0, sigma=0.04, nx=nx, ny=ny, nz=nz),
                    seed=nx + 7 * ny + nz, phi_amp=0.02)
    w.walls_z, w.stencil, w.velocity = walls, stencil, kind
    with L.Solver(w) as a, L.Solver(w, pattern="aa") as b:
        for s in (a, b):
            L.lbm_set_tuning(s.ctx, L.LBM_TUNE_BRICKS, 0)
        for n in (1, 4):
            a.step(n)
            b.step(n)
            sa, sb = a.state(), b.state()
            for k in (0, 2):  # f and phi u: the flow lattice is not used
                x, y = np.asarray(sa[k]).view(np.uint32), np.asarray(sb[k]).view(np.uint32)
                assert (x == y).all()
