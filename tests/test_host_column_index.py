"""Pull offsets of the column layout (column_index.h), compiled with g++:
every direction from every corner, face and some inner cells, on grids up to
the largest that a context takes (nx ny nz below 2^31 - 4096), gives the
wrapped neighbour's element without a 32-bit overflow on the way, shifted or, where that is said to do,
not."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1906_05448_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include "column_index.h"
static int wrap(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }
int main() {
    const int grids[][4] = {{4, 4, 1, 1}, {4, 4, 1, 16}, {4, 5, 2, 16}, {27, 26, 33, 48}, {148, 148, 438, 448},
                            {1024, 1024, 2047, 2047}, {1024, 1023, 2048, 2048}, {4, 4, 134217471, 134217471},
                            {4, 134217471, 4, 4}, {134217471, 4, 4, 4}, {46340, 46340, 1, 1}, {23170, 5792, 16, 16}};
    for (auto &g : grids) {
        const long long nx = g[0], ny = g[1], nz = g[2], zp = g[3];
        if (nx * ny * zp >= (1LL << 31) - 4096) return 9;
        const bool big = lbmgb::column_shifted((int)nx, (int)zp, nx * ny * zp);
        if (big != (nx * ny * zp + (nx + 2) * zp >= (1LL << 31))) return 8;
        for (int s = big; s < 2; s++) {  // without the shift only where it is not needed
        const long long shift = s ? lbmgb::column_shift(nx * ny * zp) : 0;
        const long long xs[] = {0, 1, nx / 2, nx - 2, nx - 1}, ys[] = {0, 1, ny / 2, ny - 2, ny - 1},
                        zs[] = {0, nz > 1 ? 1 : 0, nz / 2, nz > 1 ? nz - 2 : 0, nz - 1};
        for (long long x : xs) for (long long y : ys) for (long long z : zs)
            for (int cx = -1; cx <= 1; cx++) for (int cy = -1; cy <= 1; cy++) for (int cz = -1; cz <= 1; cz++) {
                const lbmgb::ColumnWrap w = lbmgb::column_wrap((int)x, (int)y, (int)z, (int)nx, (int)ny, (int)nz, (int)zp);
                const long long e = z + zp * (x + nx * y);
                const int o = lbmgb::column_offset((int)e - (int)shift, w, cx, cy, cz);
                const long long to = wrap((int)z - cz, (int)nz) + zp * (wrap((int)x - cx, (int)nx) + nx * wrap((int)y - cy, (int)ny));
                if (o + shift - (cz + zp * (cx + nx * cy)) != to) {
                    std::printf("%lld %lld %lld: cell %lld %lld %lld, c %d %d %d\n", nx, ny, nz, x, y, z, cx, cy, cz);
                    return 1;
                }
            }
        }
    }
    return 0;
}
"""


def test_pull_offsets_up_to_the_largest_grids(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O1", "-ftrapv", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
