"""The sizes of the randomized PROBE's level lists (csrc/rand_lists.h, plain C++): a list sized for a level takes that
level, whatever capacity an earlier call left; a capacity takes every level up to the stated one and none beyond it."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1709_06955_gb300", "csrc")
HARNESS = r"""
#include "rand_lists.h"
#include <cstdio>
using namespace ps;
static long long bad = 0;
static void check(double share, int64_t cap, int64_t E) {
    if (E < 0) return;
    const int64_t need = rand_list_entries(share, E), most = rand_list_items(share, cap);
    const bool fits = need <= cap, taken = E <= most;  // the host grows the list, or the level runs
    if (fits != taken || need > E || need > rand_list_entries(share, E + 1)) {
        if (bad++ < 10) printf("share %.17g cap %lld E %lld: sized %lld, taken up to %lld\n", share, (long long)cap,
                               (long long)E, (long long)need, (long long)most);
    }
}
int main() {
    const double shares[] = {0.125, 0.19364916731037085, 0.2, 0.25, 0.30983866769659335, 1.0 / 3, 0.5, 0.7, 0.99, 1.0};
    long long n = 0;
    for (double share : shares) {
        for (int64_t cap = 0; cap < 6000; ++cap) {  // every capacity, every E around what it holds
            const int64_t mid = (int64_t)((double)cap / share);
            for (int64_t E = mid - 24; E <= mid + 24; ++E, ++n) check(share, cap, E);
            for (int64_t E : {cap - 1, cap, cap + 1, (int64_t)1023, (int64_t)1024, (int64_t)1025}) check(share, cap, E);
        }
        for (int64_t cap = 7777; cap < (1ll << 31); cap += cap / 3 + 1) {
            const int64_t mid = (int64_t)((double)cap / share);
            for (int64_t E = mid - 40; E <= mid + 40; ++E, ++n) check(share, cap, E);
        }
        int64_t at = 0;  // a list sized for E, for every E of a range
        for (int64_t E = 0; E < 40000; ++E, ++n) check(share, at = rand_list_entries(share, E), E);
    }
    // what is refused when the two roundings are not one rule
    check(0.30983866769659335, 7794, 25152);
    check(0.125, 1152, 9209);
    check(0.25, 13071319, 52285274);
    printf("checked %lld bad %lld\n", n, bad);
    return bad != 0;
}
"""


def test_a_list_sized_for_a_level_takes_it(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "lists.cpp", tmp_path / "lists"
    src.write_text(HARNESS)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
