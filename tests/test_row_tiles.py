"""The tiles of the allocation-free residual norm's rows (csrc/row_tiles.h, the
code the kernel runs), compiled with the host compiler: every entry of 32 rows
lies in exactly one tile and the walk ends, up to entry counts of the largest
int32, where base + tile passes the last one."""

import os
import shutil
import subprocess

import pytest

from conftest import ROOT

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "row_tiles.h"
// rows of `len` entries ending at e: entries summed, tiles taken (at most 1000)
int main(int argc, char** argv) {
    const long long e = atoll(argv[1]), len = atoll(argv[2]);
    const int32_t s = (int32_t)(e - 32 * len);
    amg::RowTiles tile(s, (int32_t)e);
    long long summed = 0, tiles = 1;
    int32_t k[32];
    for (int i = 0; i < 32; ++i) k[i] = (int32_t)(s + i * len);
    for (;; ++tiles) {
        for (int i = 0; i < 32; ++i) {
            const int32_t end = tile.end_in_tile((int32_t)(s + (i + 1) * len));
            for (; k[i] < end; ++k[i], ++summed)
                if (k[i] < tile.base || k[i] - tile.base >= amg::kNaTile) return 1;
        }
        if (tiles > 1000 || !tile.next()) break;
    }
    std::printf("%lld %lld\n", summed, tiles);
}
"""


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("tiles")
    (d / "walk.cpp").write_text(SRC)
    subprocess.run([cxx, "-O1", "-std=c++17", "-fsanitize=signed-integer-overflow",
                    "-fsanitize-undefined-trap-on-error", "-I", os.path.join(ROOT, "paper_1209_0960_gb300", "csrc"),
                    str(d / "walk.cpp"), "-o", str(d / "walk")], check=True, capture_output=True)

    def run(e, length):
        out = subprocess.run([str(d / "walk"), str(e), str(length)], check=True,
                             capture_output=True, text=True).stdout
        return tuple(int(v) for v in out.split())
    return run


@pytest.mark.parametrize("length", [0, 1, 6, 7, 8, 27, 1000])
@pytest.mark.parametrize("below", [0, 1, 10, 223, 224, 225, 2**31 - 1 - 32 * 1000])
def test_every_entry_is_in_one_tile(walk, length, below):
    summed, tiles = walk(2**31 - 1 - below, length)
    assert summed == 32 * length
    assert tiles == max(1, -(-32 * length // 224))
