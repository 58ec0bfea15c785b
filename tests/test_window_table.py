"""The table of window starts, on the CPU: how many starts a list has for the sizes of an index."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = "/usr/local/cuda/include"

pytestmark = pytest.mark.skipif(not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")) or shutil.which("g++") is None,
                                reason="needs g++ and the CUDA headers")

SOURCE = r"""
#include <algorithm>
#include <cstdio>
static inline int __clz(int x) { return x ? __builtin_clz((unsigned)x) : 32; }
using std::max;
using std::min;
#include "index.cuh"
using namespace aps;

int main() {
    for (int nw : {0, 1, 2, 3, 4, 12, 100, 559, 5581, 1116072})
        for (int per : {8, 4, 1, 0})
            for (int64_t len : {0, 1, 2, 3, 10, 69, 70, 1000, 100000, 2147483647}) {
                const int s = list_shift(len, nw, per), g = window_groups(nw, s);
                // no more starts than the list has room for, and no coarser than that asks for
                if (g > 1 && g > per * len) return printf("%d %d %lld: %d groups\n", nw, per, (long long)len, g), 1;
                if (s > 0 && window_groups(nw, s - 1) <= per * len) return printf("%d %d %lld: too coarse\n", nw, per, (long long)len), 2;
                if (s > 63) return 3;
            }
    // groups cover the windows: the last one may be short
    for (int nw = 0; nw < 70; nw++)
        for (int s = 0; s < 8; s++)
            if (window_groups(nw, s) != (nw + (1 << s) - 1) / (1 << s)) return 4;
    // 200,000 rows of 50 components over 100,000 dimensions, and a million rows of 40 over 500,000: the
    // table with every window fits (W = tile_window(2))
    if (4ll * 100000 * (200000 / tile_window(2) + 2) > window_bytes(10000000, 100000)) return 5;
    if (4ll * 500000 * (1000000 / tile_window(2) + 2) > window_bytes(40000000, 500000)) return 6;
    return 0;
}
"""


def test_table_stays_in_proportion_to_the_index(tmp_path):
    src, exe = tmp_path / "t.cc", tmp_path / "t"
    src.write_text(SOURCE)
    r = subprocess.run(["g++", "-std=c++17", "-O0", "-w", "-I", CUDA, "-I", os.path.join(ROOT, "include"), "-I",
                        os.path.join(ROOT, "paper_1402_3010_gb300", "csrc"), str(src), "-o", str(exe),
                        "-Wl,--unresolved-symbols=ignore-all"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[:4000]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, (r.returncode, r.stdout)
