"""Packed pairs of transform sums in offset binary (offset_pair in csrc/ff_internal.h), checked on the CPU with the
undefined-behaviour sanitiser over the sums of half a patch (|sum| <= 8160): both halves are the sum + 32768, and adding
a second packed pair gives those of the sum of both."""
from tests.test_state_words import run_host

BODY = r"""
    const int v[] = {-8160, -8159, -257, -1, 0, 1, 255, 8159, 8160};
    int bad = 0;
    for (int lo : v)
        for (int hi : v)
            for (int lo2 : v)
                for (int hi2 : v) {
                    const int p = lo + 65536 * hi, q = lo2 + 65536 * hi2;
                    const unsigned s = ff::offset_pair(p) + (unsigned)q, d = ff::offset_pair(p) - (unsigned)q;
                    bad += (int)(s & 0xffffu) != lo + lo2 + 32768 || (int)(s >> 16) != hi + hi2 + 32768;
                    bad += (int)(d & 0xffffu) != lo - lo2 + 32768 || (int)(d >> 16) != hi - hi2 + 32768;
                }
    std::printf("%d\n", bad);
"""


def test_offset_pair(tmp_path):
    assert run_host(tmp_path, BODY) == ["0"]
