"""The listed variant of the propagation (passes of at least 300,000 pixels: candidates known not to be cheaper are
skipped, the pixels left are collected in lists).  Batches of many small ragged frames reach it with regions that are
cut by the frame on every side, in every tile shape and form; larger pairs with sub-scale grids and the extreme
search radii.  Every result is the oracle's, bit for bit; the debug-bounds build runs the same batch."""
import dataclasses
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_1805_03517_gb300 import configs
from tests import gpu_helpers as G
from tests import oracle_pins as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NAMES = ("flow_fwd", "flow_bwd", "cost_fwd", "cost_bwd", "mask")
SHAPES = [(57, 130), (64, 64), (40, 1), (2, 33), (25, 121), (7, 9), (90, 57), (17, 240), (131, 24), (49, 113)]
# tile, threads, form: regions of 32, 64 and 128 columns, tiles larger than most frames
CFGS = [(24, 16, 1, 256, 0, 0, 1), (56, 16, 1, 256, 0, 0, 2), (56, 40, 1, 512, 0, 0, 1), (120, 24, 1, 256, 0, 0, 1),
        (55, 7, 1, 512, 0, 0, 1), (24, 24, 1, 512, 0, 0, 1)]


@pytest.fixture(scope="module")
def ffm():
    from paper_1805_03517_gb300 import build, ff

    build.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return ff


def small_pairs(n):
    """n pairs of the ragged shapes: a shifted texture with a patch that moves on its own, so flows differ."""
    out = []
    for i in range(n):
        h, w = SHAPES[i % len(SHAPES)]
        a = P.smooth_texture(3000 + i, h, w)
        b = P.shifted(a, 3 - i % 7, i % 5 - 2, 4000 + i)
        if h > 30 and w > 30:
            b[10:25, 8:28] = P.smooth_texture(5000 + i, 15, 20)
        out.append((a, b))
    return out


def run_batch(ffm, pairs, prm, cfg):
    M = ffm.Matcher(prm, 0)
    if cfg is not None:
        for lvl in range(prm.n_scales):
            ffm.ff_set_tuning(M.ctx, lvl, cfg)
    dev = [(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()) for a, b in pairs]
    torch.cuda.synchronize()
    outs = M.match_frames(dev)
    M.sync()
    got = [tuple(o[k].cpu().numpy() for k in NAMES) for o in outs]
    M.close()
    return got


@pytest.mark.parametrize("T,cost,R", [(1, 0, 2), (2, 0, 2), (5, 0, 2), (3, 1, 2), (3, 0, 0), (2, 0, 16)])
def test_listed_batch_of_ragged_frames(ffm, T, cost, R):
    prm = configs.MatchParams(n_scales=2, iters=T, eps=1, rs_radius=R, cost=cost)
    pairs = small_pairs(60)
    assert 2 * sum(a.shape[0] * a.shape[1] for a, _ in pairs) > 300_000
    want = G.oracle_bidir_many(pairs, prm)
    for cfg in [None, *CFGS]:
        for g, w in zip(run_batch(ffm, pairs, prm, cfg), want):
            G.assert_same(g, w)


@pytest.mark.parametrize("sub_scales,h,w", [(1, 901, 1203), (0, 377, 641)])
def test_listed_grids_and_large_pairs(ffm, sub_scales, h, w):
    """A sub-scale grid of every second pixel that is listed itself, and a pair just past the line."""
    prm = dataclasses.replace(configs.MatchParams(n_scales=5, iters=2, eps=1), sub_scales=sub_scales)
    a = P.smooth_texture(61, h, w)
    b = P.shifted(a, 6, -4, 62)
    want = G.oracle_bidir_many([(a, b)], prm)
    G.assert_same(run_batch(ffm, [(a, b)], prm, None)[0], want[0])


CHILD = """
import os, sys
sys.path.insert(0, sys.argv[1])
from tests import test_gpu_listed as T
from tests import gpu_helpers as G
from paper_1805_03517_gb300 import configs, ff
assert ff.LIB_PATH.endswith("libff_debug.so"), ff.LIB_PATH
if __name__ == "__main__":
    pairs = T.small_pairs(60)
    for cost in (0, 1):
        prm = configs.MatchParams(n_scales=2, iters=3, cost=cost)
        want = G.oracle_bidir_many(pairs, prm)
        for cfg in [None, *T.CFGS]:
            for g, w in zip(T.run_batch(ff, pairs, prm, cfg), want):
                G.assert_same(g, w)
    print("listed debug-bounds ok")
"""


def test_listed_debug_bounds_build_runs_clean(ffm, tmp_path):
    from paper_1805_03517_gb300 import build as B

    lib = B.build(extra_flags=["-DFF_DEBUG_BOUNDS=1"], lib_path=os.path.join(B.LIBDIR, "libff_debug.so"),
                  build_dir=os.path.join(B.PKG, "_build_debug"))
    script = tmp_path / "listed_bounds.py"
    script.write_text(CHILD)
    env = dict(os.environ, FF_LIBRARY=lib, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, str(script), ROOT], env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    assert "listed debug-bounds ok" in r.stdout
