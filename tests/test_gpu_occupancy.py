"""Launches of the tile and dataflow forms fill the SMs with the variant they take: as many CTAs as its registers and
shared memory let reside, whatever the other variants'.  Under the Census cost, tile-form launches of 256 threads have
three per SM and dataflow launches of 128 threads five."""
import pytest

from paper_1805_03517_gb300 import configs
from tests import oracle_pins as P
from tests.kernel_trace import kernels
from tests.test_gpu_listed import ffm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("cost,cfg,resident,least", [
    (1, (32, 16, 1, 256, 0), False, 3), (1, (8, 8, 1, 256, 0), True, 3), (0, (32, 16, 1, 256, 0), False, 2),
    (0, (8, 8, 1, 256, 0), True, 2), (1, (32, 16, 1, 128, 0, 0, 1), False, 5), (1, (2, 4, 1, 128, 0), True, 5),
    (1, (4, 4, 1, 256, 0, 0, 1), True, 2), (0, (32, 16, 1, 128, 0, 0, 1), False, 4)])
def test_grid_fills_the_sms(ffm, tmp_path, cost, cfg, resident, least):  # noqa: F811
    h, w = 600, 800
    M = ffm.Matcher(configs.MatchParams(n_scales=5, iters=2, cost=cost), 0)
    ffm.ff_set_tuning(M.ctx, 0, cfg)
    a = P.smooth_texture(41, h, w)
    pair = [(torch.from_numpy(a).cuda(), torch.from_numpy(P.shifted(a, 3, -2, 42)).cuda())]
    torch.cuda.synchronize()
    outs = M.match_frames(pair)
    dataflow = len(cfg) > 5
    variant = f"(ff::Variant){int(resident)}" if dataflow else "true" if resident else "false"
    name = f"k_propagate{'_df' if dataflow else ''}<{cfg[3]}, ff::{'CostCensus' if cost else 'CostSad'}, {variant}>"
    found = [args for n, args in kernels(ffm, M, lambda: M.match_frames(pair, outs), tmp_path) if name in n]
    M.close()
    n_sms = torch.cuda.get_device_properties(0).multi_processor_count
    args = max(found, key=lambda args: args["grid"][0])  # of level 0
    regs = -(-args["registers per thread"] // 8) * 8
    fit = min(65536 // (regs * cfg[3]), 2048 // cfg[3], (228 << 10) // (args["shared memory"] + 1024))
    assert fit >= least, args
    tiles = 2 * -(-w // cfg[0]) * -(-h // cfg[1])
    assert args["grid"][0] == min(tiles * (2 if dataflow else 1), fit * n_sms), args
