"""The region schedule's geometry as the kernels and the plan share it (compiled
for the host, no GPU): footprint blocks, tiles, the task word, and the count of
tasks that its 32-bit positions and queue hold."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

SRC = """
#include <cstdio>
#include "aw_internal.h"
#define CHECK(c) do { if (!(c)) { printf("%s fails, S=%d\\n", #c, S); return 1; } } while (0)
int main() {
    for (int S = 2; S <= 128; ++S) {
        const int n = aw_rg_nblk(S), T = aw_rg_tile(S);
        int at = 0;
        for (int i = 0; i < n; ++i) {                       // the blocks follow one another ...
            const int w = aw_rg_blk_width(S, i);
            CHECK(aw_rg_blk_first(S, i) == at && (w == 8 || w == 16 || w == 24));
            CHECK(T + w - 1 <= AW_RG_R);                    // ... fit a region with their tile ...
            at += w;
        }
        CHECK(at == (S + 7) / 8 * 8);                       // ... and cover the padded footprint
        CHECK(n <= 8 && (16384 - S) / T < 512);             // 3 and 9 bits of the task word
        const int q = (16384 - S) / T, p = aw_rg_pack(q, q, n - 1, n - 1);
        CHECK((p & 511) == q && (p >> 9 & 511) == q && (p >> 18 & 7) == n - 1 && p >> 21 == n - 1);
    }
    const int S = 0;
    for (int npol = 1; npol <= 4; npol += 3) {
        // a queue over ntasks x npol, overshot by one a CTA (8 an SM)
        unsigned long long lim = (0xffffffffull - 8 * 1024) / npol;
        CHECK(!aw_rg_fits(lim + 8 * 1024, npol) && !aw_rg_fits(1ull << 32, npol) && !aw_rg_fits(36ull << 31, npol));
        CHECK(aw_rg_fits(1ull << 29, npol) && aw_rg_fits(0, npol));
    }
    return 0;
}
"""


def test_blocks_tiles_and_task_counts(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "geo.cc", tmp_path / "geo"
    src.write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-I" + os.path.join(ROOT, "include"), "-I" + os.path.join(CUDA, "include"),
                    "-I" + os.path.join(ROOT, "paper_2206_15117_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
