"""The rules that choose a depth's pull kernels (csrc/pull_shape.h, plain C++), which the tuner times: the tiles cover the
columns, and the tuner's matrix is one on which the level loop would take the tiles that it takes for wide depths."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1709_06955_gb300", "csrc")
HARNESS = r"""
#include "pull_shape.h"
#include <cstdio>
using namespace ps;
#define CHECK(x) \
    if (!(x)) { \
        printf("line %d: %s (n %d pieces %lld tiles %d)\n", __LINE__, #x, n, (long long)pieces, nt); \
        return 1; \
    }
int main() {
    for (int64_t n64 = 2; n64 < (1ll << 31); n64 += n64 / 5 + 1)
        for (int deg : {0, 1, 3}) {  // none, few or many pieces beside one a row
            const int32_t n = (int32_t)n64, active = deg ? n : n / 3 + 1;
            const int64_t pieces = (int64_t)active * (deg ? deg : 1);
            for (uint64_t bytes : {(uint64_t)1 << 40, (uint64_t)1 << 28, (uint64_t)0}) {
                const int32_t nt = tuner_tiles(n, pieces, active, bytes);
                const uint64_t size = 128ull * (n + 1ull) * nt;
                CHECK(nt >= 2 && nt <= 128);
                CHECK(nt == 2 || size <= std::min<uint64_t>(bytes, 1ull << 30));
                const FullTiles f = full_tiles(nt, pieces, active);
                CHECK(f.tile == (active <= kPullWideRows ? kPullWide : kPullMid) && f.per * 32 == (f.per == 4 ? 128 : 64));
                // a hundred wide tiles would be taken as such: then the tuner's tiles are, wherever there is room for them
                const bool wide = full_tiles(32 * f.per, pieces, active).wide > 0;
                if (wide && nt >= f.per && (uint64_t)128 * (n + 1) * 128 <= std::min<uint64_t>(bytes, 1ull << 30))
                    CHECK(f.wide > 0 && f.rest == 0);
                if (f.wide > 0) CHECK(full_tiles(f.per - 1, pieces, active).wide == 0);
            }
            for (int32_t nt : {0, 1, 2, 3, 4, 5, 7, 8, 31, 1000}) {
                const FullTiles f = full_tiles(nt, pieces, active);
                CHECK(f.wide * f.per + f.rest == nt && f.wide >= 0 && f.rest >= 0 && (f.wide == 0 || f.rest < f.per));
            }
        }
    return 0;
}
"""


def test_the_tuner_times_the_tiles_that_are_launched(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "shape.cpp", tmp_path / "shape"
    src.write_text(HARNESS)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
