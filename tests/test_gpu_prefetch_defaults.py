"""The default L2 prefetch distance of the stream-collide pass belongs to the kernel that runs it
(needs a GPU)."""
import pytest

from paper_1507_07294_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_1507_07294_gb300 import lbm
    lbm.load_library()
    return lbm


def _distances(L, s):
    return [L.lbm_get_tuning(s.ctx, p)
            for p in (L.LBM_TUNE_PREFETCH_COLLIDE, L.LBM_TUNE_PREFETCH_COLLIDE_SUMS)]


@pytest.mark.parametrize("pattern", ["ab", "aa"])
def test_it_follows_the_kernel_until_the_caller_sets_it(L, pattern):
    w = I.droplet(R=3.0, nx=64, ny=4, nz=4)
    with L.Solver(w, pattern=pattern) as s, L.Solver(I.droplet(R=3.0, nx=192, ny=4, nz=4), pattern=pattern) as t, \
            L.Solver(I.droplet(R=3.0, nx=33, ny=4, nz=4), pattern=pattern) as u:
        staged = _distances(L, s)
        L.lbm_set_tuning(s.ctx, L.LBM_TUNE_STENCIL_STAGE, 0)
        assert _distances(L, s) == _distances(L, t)  # two cells, rows that cannot be staged
        L.lbm_set_tuning(s.ctx, L.LBM_TUNE_CELL_PAIRS, 0)
        assert _distances(L, s) == _distances(L, u)  # one cell
        L.lbm_set_tuning(s.ctx, L.LBM_TUNE_CELL_PAIRS, 1)
        L.lbm_set_tuning(s.ctx, L.LBM_TUNE_STENCIL_STAGE, 1)
        assert _distances(L, s) == staged and staged[0] == staged[1] > 0
        assert len({staged[0], _distances(L, t)[0], _distances(L, u)[0]}) == 3
        L.lbm_set_tuning(s.ctx, L.LBM_TUNE_PREFETCH_COLLIDE, 7)
        L.lbm_set_tuning(s.ctx, L.LBM_TUNE_STENCIL_STAGE, 0)
        assert _distances(L, s) == [7, _distances(L, t)[1]]
        L.lbm_set_tuning(s.ctx, L.LBM_TUNE_PREFETCH_COLLIDE_SUMS, 9)
        L.lbm_set_tuning(s.ctx, L.LBM_TUNE_CELL_PAIRS, 0)
        assert _distances(L, s) == [7, 9]


@pytest.mark.parametrize("pattern", ["ab", "aa"])
@pytest.mark.parametrize("storage", ["fp16", "bf16"])
def test_16_bit_passes_keep_one_wave(L, storage, pattern):
    with L.Solver(I.droplet(R=3.0, nx=64, ny=4, nz=4), storage=storage, pattern=pattern) as s:
        d = _distances(L, s)
        for p in (L.LBM_TUNE_STENCIL_STAGE, L.LBM_TUNE_CELL_PAIRS):
            for v in (1, 0):
                L.lbm_set_tuning(s.ctx, p, v)
                assert _distances(L, s) == d
