"""The host rules that choose an untuned pass's variant and launch configuration (prop_listed, default_cfg), called on the
CPU from the library's own objects.  In the first iteration of a pass the listed variant has nothing to skip, so it
takes no pass of one iteration and one of two only from larger sizes on; every configuration of the default rule is one
that ff_set_tuning accepts."""
import os
import subprocess

import pytest

from paper_1805_03517_gb300 import build as B

PROGRAM = r"""
#include <cstdio>
#include "ff_internal.h"
using namespace ff;
int main() {
    for (int cost : {FF_COST_WHT_SAD, FF_COST_CENSUS})
        for (int T : {1, 2, 3, 6, 255})
            for (int df = 0; df < 2; df++)
                for (long long px = 1; px < (1ll << 33); px += 1 + px / 64) {
                    const TileCfg c = default_cfg(152, cost, px, T, df != 0);
                    const long long tiles = px / (c.tw * c.th) + 1;  // at least: of frames that are whole tiles
                    const bool listed = prop_listed(px, tiles, c.tw, c.threads, T, cost, c.dataflow > 0, 152);
                    std::printf("%d %d %d %lld %d %d %d %d %d %d %d %d\n", cost, T, df, px, c.tw, c.th, c.k, c.threads,
                                c.cluster, c.dataflow, (int)listed,
                                (int)(prop_threads_ok(c.threads) && prop_smem_bytes(c.tw, c.th, c.k) <= kMaxPropSmem));
                }
    return 0;
}
"""


def run(program, d):
    """The lines of numbers a main() linked with the library's objects prints."""
    B.build()
    src, exe = d / "rules.cu", d / "rules"
    src.write_text(program)
    objs = [os.path.join(B.BUILD, s.replace(".cu", ".o")) for s in B.SOURCES]
    r = subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-o", str(exe), str(src), *objs], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    return [tuple(int(v) for v in line.split()) for line in out.splitlines()]


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    return run(PROGRAM, tmp_path_factory.mktemp("rules"))


def test_default_configurations_are_valid(rows):
    for cost, T, df, px, tw, th, k, threads, cluster, dataflow, listed, fits in rows:
        assert fits and 1 <= k <= T and cluster == 0 and dataflow in (0, 1), (cost, T, df, px)
        assert not dataflow or (df and k == 1 and tw >= 4 and th >= 4), (cost, T, df, px)
        assert not listed or dataflow, (cost, T, df, px)


def test_listed_variant_by_iterations(rows):
    for cost, T, df, px, *_, dataflow, listed, _ in rows:
        least = {1: None, 2: 1_200_000 if cost else None}.get(T, 300_000)
        assert listed == int(bool(df) and least is not None and px >= least), (cost, T, df, px)


def test_few_census_iterations_take_the_tile_form(rows):
    """Its direct kernel has three CTAs per SM under the Census cost, the dataflow form's has two."""
    for cost, T, df, px, *_, dataflow, listed, _ in rows:
        if cost == 1 and (T == 1 or (T == 2 and not listed and (px <= 130_000 or px >= 300_000))):
            assert not dataflow, (T, df, px)


@pytest.mark.parametrize("cost,T,px,tile", [(0, 3, 892_928, (56, 16)), (0, 6, 892_928, (56, 16)), (0, 3, 700_000, (24, 24)),
                                            (1, 3, 446_464, (24, 24)), (1, 6, 465_750, (24, 24)), (0, 6, 320_000, (24, 16)),
                                            (1, 6, 320_000, (24, 16)), (1, 6, 620_000, (56, 16))])
def test_listed_tiles(rows, cost, T, px, tile):
    """Passes of a size at which 24x16 tiles were measured slower than the former rule take larger ones."""
    near = min((r for r in rows if r[0] == cost and r[1] == T and r[2]), key=lambda r: abs(r[3] - px))
    assert (near[4], near[5]) == tile and near[10], near


# pixels, tiles, tile width, threads, iterations -> listed
CASES = [((465_750, 198, 56, 256, 3), 0), ((465_750, 198, 56, 256, 6), 0), ((465_750, 198, 56, 256, 10), 1),
         ((465_750, 607, 24, 256, 9), 0), ((465_750, 608, 24, 256, 3), 1), ((465_750, 303, 24, 512, 6), 0),
         ((465_750, 304, 24, 512, 6), 1), ((2_073_600, 720, 120, 256, 5), 0), ((2_073_600, 720, 120, 256, 6), 1),
         ((2_073_600, 2000, 64, 256, 6), 0), ((2_073_600, 2000, 56, 128, 6), 0), ((299_999, 2000, 24, 256, 6), 0),
         ((2_073_600, 1575, 56, 256, 2), 0)]


def test_listed_variant_by_tiles(tmp_path):
    """It has twice the direct variant's CTAs, which fewer tiles leave idle, unless enough iterations are skipped."""
    calls = "".join("    std::printf(\"%%d\\n\", (int)prop_listed(%d, %d, %d, %d, %d, 0, true, 152));\n" % c for c, _ in CASES)
    got = run('#include <cstdio>\n#include "ff_internal.h"\nusing namespace ff;\nint main() {\n' + calls + "}\n", tmp_path)
    assert [g[0] for g in got] == [want for _, want in CASES]


FIT = r"""
#include <cstdio>
#include "ff_internal.h"
using namespace ff;
int main() {
    long long n = 0, shrunk = 0, bad = 0;
    for (int tw = 4; tw <= 1024; tw++)
        for (int th = 4; th <= 1024; th++) {
            if (prop_smem_bytes(tw, th, 1) > kMaxPropSmem) continue;  // ff_set_tuning refuses it
            int w = tw, h = th, slots = 4;
            prop_fit_tile(w, h);
            while (2 * slots < w + 2 * kHaloPerIter) slots *= 2;
            n++;
            shrunk += w != tw || h != th;
            bad += w > tw || h > th || w < 4 || h < 4 || prop_launch_smem(w, h, 1, true) > kMaxTileSmem ||
                   slots * (h + 2 * kHaloPerIter + 2) > 8192;  // a list entry has 13 bits for the slot
        }
    std::printf("%lld %lld %lld\n", n, shrunk, bad);
    return 0;
}
"""


def test_every_tile_fits_the_listed_variant(tmp_path):
    n, shrunk, bad = run(FIT, tmp_path)[0]
    accepted = sum(8 * (tw + 8) * (th + 8) <= 200 * 1024 for tw in range(4, 1025) for th in range(4, 1025))
    assert n == accepted and 0 < shrunk < n and bad == 0
