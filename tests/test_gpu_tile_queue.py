"""The queue of the tile form: CTA b starts with entry b, further entries are taken with a counter, and a launch with a
CTA per tile takes none.  Launches with fewer tiles than the GPU has CTAs, about as many, and many times more, with
whole and cut tiles; every result is the oracle's, bit for bit."""
import pytest

from paper_1805_03517_gb300 import configs
from tests import gpu_helpers as G
from tests import oracle_pins as P
from tests.test_gpu_listed import ffm, run_batch  # noqa: F401  (ffm: fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_scales,h,w", [(1, 31, 45), (3, 96, 128), (4, 187, 250)])
@pytest.mark.parametrize("cfg", [(8, 4, 1, 256, 0), (8, 4, 2, 512, 0), (5, 7, 3, 128, 0), (32, 32, 1, 256, 0)])
@pytest.mark.parametrize("cost", [0, 1])
def test_tile_queue(ffm, n_scales, h, w, cfg, cost):  # noqa: F811
    prm = configs.MatchParams(n_scales=n_scales, iters=3, eps=1, cost=cost)
    a = P.smooth_texture(71, h, w)
    b = P.shifted(a, 2, -1, 72)
    want = G.oracle_bidir_many([(a, b)], prm)
    for _ in range(2):  # the second run finds the counter as the first left it
        G.assert_same(run_batch(ffm, [(a, b)], prm, cfg)[0], want[0])
