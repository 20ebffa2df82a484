"""The stamps of the listed variant's state words (still_concerned in csrc/ff_internal.h), checked on the CPU with the
undefined-behaviour sanitiser: for the stamps a task writes (0..8), the neighbours that have not tried the pixel since
the stamped half-sweep, recomputed here from the schedule; nobody for the other values a 4-bit field can hold, which a
task reads after a wait that expired."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1805_03517_gb300", "csrc")


def run_host(tmp_path, body):
    """Compiles a main() over ff_internal.h for the host, runs it and returns its lines; undefined behaviour fails."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "host.cu", tmp_path / "host"
    src.write_text('#include <cstdio>\n#include "ff_internal.h"\nint main() {\n' + body + "\n    return 0;\n}\n")
    r = subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler",
                        "-fsanitize=undefined,-fno-sanitize-recover=all", "-I", os.path.join(ROOT, "include"), "-I",
                        CSRC, "-o", str(exe), str(src)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return r.stdout.splitlines()


def expected(stamp):
    """Bits (right, left, below, above) of the neighbours whose last trial of the pixel came before its change."""
    if not 1 <= stamp <= 8:
        return 0
    j = stamp - 1
    k = 1 - j % 2  # the neighbours' colour: they are updated in the half-sweeps 2d + k of directions d
    sides = [(0, 2), (1, 3), (0, 1), (2, 3)]  # directions in which the pixel right / left / below / above tries it
    return sum(1 << i for i, dirs in enumerate(sides) if max(2 * d + k for d in dirs) < j)


def test_stamps(tmp_path):
    lines = run_host(tmp_path, '    for (unsigned s = 0; s < 16; s++) std::printf("%u\\n", ff::still_concerned(s));')
    assert [int(v) for v in lines] == [expected(s) for s in range(16)]
