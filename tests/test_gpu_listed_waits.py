"""The bounded waits of the listed variant: with the tiles' progress withheld every wait of its launches expires, in the
queue and in the affine variant, and its tasks go on with whatever the buffers hold: plain costs and state words of the
context's earlier calls, under either cost.  ff_sync reports FF_ERR_TIMEOUT, and the same context then matches
bit-exactly again."""
import pytest

from paper_1805_03517_gb300 import configs
from tests import gpu_helpers as G
from tests import oracle_pins as P
from tests.test_gpu_listed import NAMES, ffm  # noqa: F401  (ffm: fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dataflow,cost", [(1, 0), (2, 0), (1, 1)])
def test_expired_waits_are_reported_and_the_context_recovers(ffm, dataflow, cost):  # noqa: F811
    prm = configs.MatchParams(n_scales=4, iters=3, eps=1, cost=cost)
    h, w = 375, 500
    assert 2 * h * w > 300_000  # level 0 is listed
    a = P.smooth_texture(700, h, w)
    b = P.shifted(a, 5, -3, 701)
    M = ffm.Matcher(prm, 0)
    ffm.ff_set_option(M.ctx, ffm.FF_OPT_SEED_KERNEL, ffm.FF_SEED_MMA_SYNC)  # only the propagation waits
    ffm.ff_set_tuning(M.ctx, 0, (24, 16, 1, 256, 0, 0, dataflow))
    pair = (torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda())
    torch.cuda.synchronize()
    want = G.oracle_bidir_many([(a, b)], prm)[0]

    def match():
        out = M.match_frames([pair])[0]
        M.sync()
        return tuple(out[k].cpu().numpy() for k in NAMES)

    G.assert_same(match(), want)
    ffm.ff_set_option(M.ctx, ffm.FF_OPT_WAIT_LIMIT, 2000)
    ffm.ff_set_option(M.ctx, ffm.FF_OPT_TEST_WITHHOLD_COPIES, 1)  # no tile publishes its progress
    with pytest.raises(ffm.FFError) as e:
        match()
    assert e.value.status == ffm.FF_ERR_TIMEOUT
    assert "dataflow" in str(e.value)
    ffm.ff_set_option(M.ctx, ffm.FF_OPT_TEST_WITHHOLD_COPIES, 0)
    ffm.ff_set_option(M.ctx, ffm.FF_OPT_WAIT_LIMIT, 1 << 22)
    G.assert_same(match(), want)
    M.close()
