"""Which frames fit the fixed scratch of ff_match_pair_noalloc is part of its interface: the flows, the tables and the
queues of the compact configurations decide, not those of the configurations the call runs for speed.  The largest
frame that fits (where only the compact configurations do) matches like ff_match_pair, bit for bit; one with two rows more
is refused."""
import pytest

from paper_1805_03517_gb300 import configs
from tests import oracle_pins as P
from tests.test_gpu_listed import ffm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
LIMIT = 32 << 20


def scratch_bytes(w, h, L, T, n_sms):
    """Bytes the call needs with the compact configurations (up to 1.5 KB of small tables)."""
    up = lambda n: -(-n // 256) * 256  # noqa: E731
    total, launches = 1024, 0
    for s in range(L):
        ws, hs = w >> s, h >> s
        n = ws * hs
        tw, th, k = ((32, 32, 1) if n // 1024 >= 4 * n_sms else (32, 16, 1) if n // 512 >= 4 * n_sms
                     else (16, 16, min(2, T)) if n // 256 >= 2 * n_sms else (8, 8, min(3, T)))
        launches += -(-T // k)
        total += up(8 * -(-ws // tw) * -(-hs // th)) + 4 * up(4 * n)
    return total + up(4 * (w >> (L - 1)) * (h >> (L - 1))) + up(120 * launches) + up(4 * launches)


@pytest.mark.parametrize("T", [6, 96])
def test_largest_frame(ffm, T):  # noqa: F811
    n_sms = torch.cuda.get_device_properties(0).multi_processor_count
    w, L = 256, 5
    prm = configs.MatchParams(n_scales=L, iters=T, eps=1)
    h = next(h for h in range(8192, 0, -1) if scratch_bytes(w, h, L, T, n_sms) + 1536 <= LIMIT)
    M = ffm.Matcher(prm, 0)
    for rows, fits in ((h, True), (h + 2, False)):
        a = P.smooth_texture(51, rows, w)
        X, Y = (M.features(torch.from_numpy(i).cuda()) for i in (a, P.shifted(a, 3, -2, 52)))
        flow = torch.full((rows, w, 2), -7, dtype=torch.int16, device="cuda")
        cost = torch.full((rows, w), -7, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        if fits:
            ffm.ff_match_pair_noalloc(M.ctx, X.handle, Y.handle, 0, flow.data_ptr(), cost.data_ptr())
            M.sync()
            want_flow, want_cost = M.match_pair(X, Y, 0)
            M.sync()
            assert torch.equal(flow, want_flow) and torch.equal(cost, want_cost)
        else:
            with pytest.raises(ffm.FFError):
                ffm.ff_match_pair_noalloc(M.ctx, X.handle, Y.handle, 0, flow.data_ptr(), cost.data_ptr())
        M.release(X)
        M.release(Y)
    M.close()
