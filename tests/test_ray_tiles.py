"""The tiles of rays whose sample counts are totalled together: over every batch size that
a step or a render accepts, each tile's totals are cleared by exactly one thread of the ray
generation and no thread clears anything behind them.  The predicate the kernels use is
compiled for the host and walked over all threads of the launch (no GPU needed)."""

import os
import subprocess

from paper_2210_13641_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "rays.cuh"

int main(int argc, char** argv) {
    for (int a = 1; a < argc; ++a) {
        const uint32_t n = (uint32_t)strtoul(argv[a], nullptr, 10), threads = (n + 255u) / 256u * 256u;
        uint32_t cleared = 0, last = 0;
        for (uint32_t i = 0; i < threads; ++i)
            if (nm::clears_tile(i, n)) {
                ++cleared;
                last = i;
            }
        printf("%u %u %u\n", n, cleared, last);
    }
    return 0;
}
"""

T = 4096
SIZES = [1, 255, T - 1, T, T + 1, 2 * T, (1 << 20) - 1, 1 << 20, (1 << 20) + 1, (1 << 20) + T + 1, 1 << 21,
         3 * (1 << 21) + 5, (1 << 24) - 1, 1 << 24]


def test_totals_of_exactly_the_batch_tiles_are_cleared(tmp_path):
    src, exe = tmp_path / "tiles.cu", tmp_path / "tiles"
    src.write_text(PROGRAM)
    p = subprocess.run([build._nvcc(), build.ARCH, "-std=c++17", "-O2", "-I", build.CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert p.returncode == 0, p.stderr
    r = subprocess.run([str(exe)] + [str(n) for n in SIZES], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    rows = [tuple(map(int, line.split())) for line in r.stdout.splitlines()]
    assert rows == [(n, (n + T - 1) // T, (n + T - 1) // T - 1) for n in SIZES]
