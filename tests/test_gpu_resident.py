"""The resident variant of the propagation (regions of at most one pixel per thread): every thread count and form, a
region of exactly a pixel per thread, regions of odd width, frames smaller than a tile and frames that cut tiles on
every side, one to three iterations per launch, extreme search radii, sub-scale grids.  Every result is the oracle's,
bit for bit."""
import pytest

from paper_1805_03517_gb300 import configs
from tests import gpu_helpers as G
from tests import oracle_pins as P
from tests.test_gpu_listed import ffm, run_batch  # noqa: F401  (ffm: fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
# tile, iterations per launch, threads, form; the regions have 120, 256 (all threads), 255 in rows of 17, 480, 480 and
# 192 pixels
CFGS = [(2, 4, 1, 128, 0), (8, 8, 1, 256, 0), (9, 7, 1, 512, 0), (8, 4, 2, 512, 0), (16, 12, 1, 512, 0, 0, 1),
        (4, 8, 1, 256, 0, 0, 2)]


@pytest.mark.parametrize("cfg", CFGS + [None])
@pytest.mark.parametrize("T,cost,R,sub", [(1, 0, 2, 0), (5, 0, 2, 0), (4, 1, 2, 0), (3, 0, 0, 0), (3, 0, 16, 0), (3, 0, 2, 1)])
def test_resident(ffm, cfg, T, cost, R, sub):  # noqa: F811
    prm = configs.MatchParams(n_scales=3, iters=T, eps=1, rs_radius=R, cost=cost, sub_scales=sub)
    pairs = []
    for i, (h, w) in enumerate([(33, 50), (64, 96), (97, 61), (9, 11)]):
        a = P.smooth_texture(81 + i, h, w)
        b = P.shifted(a, 2 - i, i - 1, 91 + i)
        if h > 30:
            b[8:20, 10:25] = P.smooth_texture(95 + i, 12, 15)
        pairs.append((a, b))
    for pair in pairs:
        want = G.oracle_bidir_many([pair], prm)
        G.assert_same(run_batch(ffm, [pair], prm, cfg)[0], want[0])
