"""Scratch of the spectra (spectra_scratch.h), compiled with g++: whatever the
entry point lets through fits the population buffer, for every cube side,
storage size and number of bins, and keeps at least one block."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1906_05448_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include "spectra_scratch.h"
int main() {
    long long accepted = 0, fewer = 0;
    for (int n = 8; n <= 1024; n *= 2)
        for (int sb = 2; sb <= 8; sb *= 2)
            for (int q = 19; q <= 27; q += 8)
                for (int nbins = 1; nbins <= 2048; nbins++) {
                    const long long N = (long long)n * n * n;
                    if (lbmgb::spectrum_scratch_bytes(N, nbins) > 19 * (size_t)N * sb) continue;
                    accepted++;
                    const size_t buffer = (size_t)q * N * sb;
                    const int pairs = n <= 8 ? 4 : (n <= 256 ? 8 : 4);
                    const int b = lbmgb::spectrum_blocks(buffer, N, n, pairs, nbins, 1 << 20);
                    if (b < 1 || b > lbmgb::SP_BLOCKS) return 1;
                    if (lbmgb::spectrum_bins_offset(N) + 16 * (size_t)nbins * b > buffer) return 2;
                    long long all = (long long)n * (n / 2) / pairs;
                    if (all > lbmgb::SP_BLOCKS) all = lbmgb::SP_BLOCKS;
                    if (b < all) fewer++;
                    if (b < 200 && b < all) return 3;
                }
    std::printf("%lld %lld\n", accepted, fewer);
    return 0;
}
"""


def test_layout_fits_what_the_call_accepts(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.returncode
    accepted, fewer = map(int, r.stdout.split())
    assert accepted > 20000
    assert fewer > 0  # the case the limit of the call alone does not cover: 64^3 in 16 bits with 1409 bins or more
