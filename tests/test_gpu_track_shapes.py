"""Which kernels the tracking step (pattern AB, FP32) takes by the shape of the grid, each at its
edges and on both sides of the lines between them, against the three passes of the in-place
pattern (needs a GPU)."""
import numpy as np
import pytest

from paper_1507_07294_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_1507_07294_gb300 import lbm
    lbm.load_library()
    return lbm


def _workload(shape, walls, kind=("deformation", 0.02, 50.0), stencil="d3q15"):
    w = I.droplet(n=4, R=1.0, D=2.0, sigma=0.04)
    w.nx, w.ny, w.nz = shape
    w.walls_z, w.velocity, w.stencil = walls, kind, stencil
    w.phi0 = np.random.default_rng(sum(shape)).uniform(-1.0, 1.0, shape[::-1])
    return w


def _compare(L, w, one_pass):
    with L.Solver(w) as a, L.Solver(w, pattern="aa") as b:
        for s in (a, b):
            L.lbm_set_tuning(s.ctx, L.LBM_TUNE_BRICKS, 0)
        L.lbm_profile(a.ctx, True)
        for n in (1, 3):
            a.step(n)
            b.step(n)
            sa, sb = a.state(), b.state()
            for k in (0, 2):  # f and phi u: the flow lattice is not used
                assert np.array_equal(sa[k].view(np.uint32), sb[k].view(np.uint32))
        assert L.lbm_profile_read(a.ctx, L.KERNEL_PHI)[1] == (0 if one_pass else 4)
        assert L.lbm_profile_read(a.ctx, L.KERNEL_COLLIDE)[1] == 4


# as many blocks of 8 rows and 32 planes as SMs, columns and segments full and not; few planes
@pytest.mark.parametrize("kind,walls,stencil", [(("deformation", 0.02, 50.0), False, "d3q15"),
                                                (("rotation", 0.001), True, "d3q15"),
                                                (("uniform", 0.02), True, "d3q7")])
@pytest.mark.parametrize("shape", [(160, 17, 340), (1024, 9, 70), (1024, 5, 150), (992, 8, 161),
                                   (64, 40, 512), (32, 1, 1), (96, 17, 8), (32, 9, 3)])
def test_columns(L, shape, walls, kind, stencil):
    _compare(L, _workload(shape, walls, kind, stencil), True)


# tile rows with too few blocks for columns, or columns of at most 4 rows; other rows
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("shape", [(32, 32, 32), (32, 33, 9), (64, 4, 400), (32, 1, 40), (160, 5, 2000),
                                   (8, 4, 700), (33, 17, 70), (3, 3, 9), (1, 2000, 1)])
def test_bricks(L, shape, walls):
    _compare(L, _workload(shape, walls), True)


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("shape", [(1, 1, 26000), (2, 1, 52000), (3, 3, 240000), (32, 1, 30000)])
def test_thin_grids_take_three_passes(L, shape, walls):
    _compare(L, _workload(shape, walls), False)
