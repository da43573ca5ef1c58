"""The queue's tile and pair orders (tiles.cuh, compiled for the host): every
tile of a triangle or a block grid once and inside it, and the line of an entry
for triangles of up to 2^61 entries."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
HEADER = os.path.join(os.path.dirname(HERE), "paper_2404_07183_gb300", "csrc", "tiles.cuh")

SOURCE = r'''
#include "%s"
#include <cstdio>
#include <random>
#include <vector>
using namespace pcfgb;
int main()
{
    long bad = 0, seen_tiles = 0;
    for (int64_t n = 1; n <= 130; ++n) {
        const int64_t total = n * (n + 1) / 2;
        for (int order = 0; order < 2; ++order) {
            std::vector<char> seen(n * n, 0);
            for (int64_t t = 0; t < total; ++t) {
                int64_t bi = -1, bj = -1;
                decode_upper_tile(n, t, order, bi, bj);
                if (bi < 0 || bj < bi || bj >= n || seen[bi * n + bj]++) ++bad;
                ++seen_tiles;
            }
        }
        int64_t t = 0;
        for (int64_t m = 0; m < n; ++m)
            for (int64_t q = 0; q < n - m; ++q, ++t) bad += upper_line(n, t) != m;
    }
    for (int64_t r = 1; r <= 50; ++r)
        for (int64_t c = 1; c <= 50; ++c) {
            std::vector<char> seen(r * c, 0);
            for (int64_t t = 0; t < r * c; ++t) {
                int64_t bi = -1, bj = -1;
                decode_cross_tile(r, c, t, bi, bj);
                if (bi < 0 || bi >= r || bj < 0 || bj >= c || seen[bi * c + bj]++) ++bad;
            }
        }
    std::mt19937_64 g(1);
    for (int64_t n : {(int64_t)65535, (int64_t)65536, (int64_t)92682, (int64_t)92683, (int64_t)1048583,
                      (int64_t)0x7fffffff}) {
        auto start = [n](int64_t m) { return m * n - m * (m - 1) / 2; };
        auto check = [&](int64_t m) {
            bad += upper_line(n, start(m)) != m;
            bad += upper_line(n, start(m) + (n - m) - 1) != m;
            bad += upper_line(n, start(m) + (int64_t)(g() %% (uint64_t)(n - m))) != m;
        };
        for (int64_t m = 0; m < 2000; ++m) { check(m); check(n - 1 - m); }
        for (int i = 0; i < 20000; ++i) check((int64_t)(g() %% (uint64_t)n));
    }
    printf("%%ld %%ld\n", seen_tiles, bad);
    return 0;
}
'''


def test_every_tile_once(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE % HEADER)
    subprocess.run([gxx, "-O1", "-o", str(exe), str(src)], check=True)
    tiles, bad = map(int, subprocess.run([str(exe)], capture_output=True, text=True,
                                         check=True).stdout.split())
    assert tiles == 2 * sum(n * (n + 1) // 2 for n in range(1, 131)) and bad == 0
