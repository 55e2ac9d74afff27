"""The sizes a build chooses by itself (csrc/build_sizes.h), compiled here with
g++, and that the autotuner's answer is not worse than no answer."""
import shutil
import subprocess
from pathlib import Path

import numpy as np
import pytest

from paper_1304_4661_gb300 import graphgen as gg
from paper_1304_4661_gb300 import pll

ROOT = Path(__file__).resolve().parents[1]

CHECK = r"""
#include <cstdio>
#include "build_sizes.h"
using namespace pll;
int main() {
    const uint32_t ns[] = {1, 4096, 16384, 16385, 32768, 32769, 573000, (1u << 24) - 1};
    for (uint32_t n : ns)
        for (uint32_t d = 1024; d <= BATCH_MAX; d *= 2) {
            uint32_t s[7];
            const int c = autotune_batches(n, d, s);
            for (int i = 0; i < c; ++i) printf("%u%c", s[i], i + 1 < c ? ' ' : ';');
        }
    printf("\n");
    const uint64_t gb = 1ull << 30;
    printf("%llu %llu %llu %llu\n", (unsigned long long)slice_entries(10, 280 * gb),
           (unsigned long long)slice_entries(31000000, 280 * gb), (unsigned long long)slice_entries(4000000000ull, 280 * gb),
           (unsigned long long)slice_entries(4000000000ull, 0));
}
"""


def test_sizes(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not available")
    (tmp_path / "c.cpp").write_text(CHECK)
    subprocess.run([gxx, "-std=c++17", "-Wall", "-Werror", f"-I{ROOT / 'paper_1304_4661_gb300' / 'csrc'}",
                    str(tmp_path / "c.cpp"), "-o", str(tmp_path / "c")], check=True)
    tried, slices = subprocess.run([tmp_path / "c"], capture_output=True, text=True, check=True).stdout.splitlines()
    tried = iter([int(x) for x in s.split()] for s in tried.split(";")[:-1])
    base = [1024, 2048, 4096, 8192, 16384]
    for n in (1, 4096, 16384, 16385, 32768, 32769, 573000, (1 << 24) - 1):
        for default in (1024, 2048, 4096, 8192, 16384, 32768, 65536):
            more = [b for b in (32768, 65536) if b <= default and b // 2 < n]
            assert next(tried) == base + more, (n, default)
    assert slices.split() == [str(1 << 16), "31000000", str(64 << 20), str(1 << 16)]


@pytest.mark.gpu
def test_the_autotuner_looks_at_the_default():
    """1500 small graphs in one build: 65536 roots a batch (the default) take 3.9 ms, 16384 5.0 ms."""
    from .gpu_util import dev_u32
    off, col, start = gg.union([gg.ba(100, 3, i) for i in range(1500)])
    rb, block, ms = pll.autotune(dev_u32(off), dev_u32(col), 4, graph_start=np.asarray(start))
    assert rb > 16384 and block in (128, 256, 512) and ms > 0
