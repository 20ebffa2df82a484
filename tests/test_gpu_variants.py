"""Which variant of the propagation a pass takes, seen in a trace of the kernels, and that its results are the oracle's.
The listed variant: batches of ragged frames with ten iterations (any number of tiles) in every tile shape, tiles that
have to be shrunk to what it can hold (one by its bytes, two by its slots), both costs and the extreme search radii;
passes just below and above its sizes with one to three iterations.  The debug-bounds build runs the shrunk tiles too."""
import os
import subprocess
import sys

import pytest

from paper_1805_03517_gb300 import configs
from tests import gpu_helpers as G
from tests import oracle_pins as P
from tests import test_gpu_listed as TL
from tests.kernel_trace import kernels
from tests.test_gpu_listed import ffm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
LISTED, DIRECT = "(ff::Variant)2>", "(ff::Variant)0>"
SHRUNK = [(120, 180, 1, 256, 0, 0, 1), (4, 1024, 1, 256, 0, 0, 1), (1000, 12, 1, 512, 0, 0, 2)]


def run_traced(ffm, pairs, prm, cfg, tmp_path):  # noqa: F811
    """The outputs of the batch and the names of the propagation kernels that made them."""
    M = ffm.Matcher(prm, 0)
    for lvl in range(prm.n_scales if cfg else 0):
        ffm.ff_set_tuning(M.ctx, lvl, cfg)
    dev = [(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()) for a, b in pairs]
    torch.cuda.synchronize()
    outs = M.match_frames(dev)
    names = [n for n, _ in kernels(ffm, M, lambda: M.match_frames(dev, outs), tmp_path) if "k_propagate" in n]
    got = [tuple(o[k].cpu().numpy() for k in TL.NAMES) for o in outs]
    M.close()
    return got, names


@pytest.mark.parametrize("cost,R", [(0, 2), (1, 2), (0, 0), (0, 16)])
def test_listed_batch(ffm, tmp_path, cost, R):  # noqa: F811
    prm = configs.MatchParams(n_scales=2, iters=10, eps=1, rs_radius=R, cost=cost)
    pairs = TL.small_pairs(60)
    want = G.oracle_bidir_many(pairs, prm)
    for cfg in [None, *TL.CFGS, *SHRUNK]:
        got, names = run_traced(ffm, pairs, prm, cfg, tmp_path)
        assert LISTED in names[-1] and "k_propagate_df" in names[-1], (cfg, names)  # level 0
        for g, w in zip(got, want):
            G.assert_same(g, w)


@pytest.mark.parametrize("n,h,w,T,last", [(1, 374, 401, 3, DIRECT), (1, 375, 401, 3, LISTED), (1, 375, 401, 2, DIRECT),
                                          (1, 375, 401, 1, "k_propagate<"), (4, 375, 401, 2, DIRECT)])
def test_line_between_the_variants(ffm, tmp_path, n, h, w, T, last):  # noqa: F811
    """Passes of 299,948 and 300,750 pixels, and of four times as many."""
    check_line(ffm, tmp_path, n, h, w, configs.MatchParams(n_scales=4, iters=T, eps=1), last)


@pytest.mark.parametrize("n,h,w,T,last", [(1, 374, 401, 3, DIRECT), (1, 375, 401, 3, LISTED), (1, 375, 401, 2, "k_propagate<"),
                                          (4, 374, 401, 2, "k_propagate<"), (4, 375, 401, 2, LISTED)])
def test_line_between_the_variants_census(ffm, tmp_path, n, h, w, T, last):  # noqa: F811
    check_line(ffm, tmp_path, n, h, w, configs.MatchParams(n_scales=4, iters=T, eps=1, cost=1), last)


def check_line(ffm, tmp_path, n, h, w, prm, last):  # noqa: F811
    pairs = []
    for i in range(n):
        a = P.smooth_texture(800 + i, h, w)
        pairs.append((a, P.shifted(a, 5 - i, i - 3, 810 + i)))
    got, names = run_traced(ffm, pairs, prm, None, tmp_path)
    assert last in names[-1], names
    for g, w_ in zip(got, G.oracle_bidir_many(pairs, prm)):
        G.assert_same(g, w_)


CHILD = """
import sys
sys.path.insert(0, sys.argv[1])
from tests import test_gpu_listed as TL, test_gpu_variants as T
from tests import gpu_helpers as G
from paper_1805_03517_gb300 import configs, ff
assert ff.LIB_PATH.endswith("libff_debug.so"), ff.LIB_PATH
if __name__ == "__main__":
    prm = configs.MatchParams(n_scales=2, iters=10, eps=1)
    pairs = TL.small_pairs(60)
    want = G.oracle_bidir_many(pairs, prm)
    for cfg in [*TL.CFGS, *T.SHRUNK]:
        for g, w in zip(TL.run_batch(ff, pairs, prm, cfg), want):
            G.assert_same(g, w)
    print("variants debug-bounds ok")
"""


def test_debug_bounds_build_runs_clean(ffm, tmp_path):  # noqa: F811
    from paper_1805_03517_gb300 import build as B

    lib = B.build(extra_flags=["-DFF_DEBUG_BOUNDS=1"], lib_path=os.path.join(B.LIBDIR, "libff_debug.so"),
                  build_dir=os.path.join(B.PKG, "_build_debug"))
    script = tmp_path / "variants_bounds.py"
    script.write_text(CHILD)
    env = dict(os.environ, FF_LIBRARY=lib, PYTHONPATH=TL.ROOT)
    r = subprocess.run([sys.executable, str(script), TL.ROOT], env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    assert "variants debug-bounds ok" in r.stdout
