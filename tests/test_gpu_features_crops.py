"""Descriptors of crops: frames whose first byte and whose rows lie on any byte, wide enough (71 pixels and more) for
tiles staged from aligned words.  Every level equals the oracle's of the same pixels, with the single and the batched
call and with Census patterns, also for frames of only 0 and 255, whose sums are the largest."""
import numpy as np
import pytest

from paper_1805_03517_gb300 import configs
from tests import oracle_pins as P
from tests.test_gpu_listed import ffm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("x0", [0, 1, 2, 3])
@pytest.mark.parametrize("w", [70, 71, 72, 103, 200])
def test_crops(ffm, orc, w, x0):  # noqa: F811
    h, y0, pad = 37, 2, (w + x0) % 3  # rows of 3 * (w + x0 + pad) bytes, the last one ending the allocation if pad is 0
    big = P.rand_img(900 + w + x0, h + y0, w + x0 + pad)
    if x0 & 1:
        big = np.where(big < 128, 0, 255).astype(np.uint8)
    img = np.ascontiguousarray(big[y0:, x0:x0 + w])
    M = ffm.Matcher(configs.MatchParams(n_scales=3, iters=1, cost=1), 0)
    dev = torch.from_numpy(big).cuda()[y0:, x0:x0 + w]
    torch.cuda.synchronize()
    for pyr in (M.features(dev), M.features_batch([dev, dev])[1]):
        for s, lv in enumerate(orc.pyramid(img, 3)):
            got, cen = M.level_features(pyr, s), M.level_census(pyr, s)
            M.sync()
            assert np.array_equal(got.cpu().numpy(), orc.wht(lv)), (w, x0, s)
            assert np.array_equal(cen.cpu().numpy().astype(np.uint64), orc.census(lv)), (w, x0, s)
    M.close()
