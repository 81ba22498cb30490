// Scratch of the spectra (spectra.cu) in the population buffer that the next
// step overwrites: two complex FP32 fields (16 bytes per cell), then the
// shell sums of each block of the last pass (2 nbins doubles). Host code
// without CUDA, so that the layout is checked on the CPU.
#pragma once

#include <stddef.h>

namespace lbmgb {

constexpr int SP_BLOCKS = 304;  // blocks of the z pass that own a set of bins, at most

// what the call asks of the buffer (a limit of the ABI: calls beyond it answer LBM_ENOMEM)
inline size_t spectrum_scratch_bytes(long long N, int nbins) {
    return ((size_t)N * 8 + 255) / 256 * 256 + sizeof(double) * 2 * (size_t)nbins * 304;
}

inline size_t spectrum_bins_offset(long long N) { return 16 * (size_t)N; }

// Blocks of the z pass: as many as run together, have work (n n/2 pairs of
// lines, `pairs` to a block) and have room for their bins. The limit above
// counts one field and 304 sets of bins, so a call that it lets through has
// room behind both fields for 223 sets or more.
inline int spectrum_blocks(size_t buffer, long long N, int n, int pairs, int nbins, int resident) {
    const size_t room = buffer > spectrum_bins_offset(N)
                            ? (buffer - spectrum_bins_offset(N)) / (sizeof(double) * 2 * (size_t)nbins) : 0;
    long long b = resident < 1 ? 1 : resident;
    if (b > SP_BLOCKS) b = SP_BLOCKS;
    if (b > (long long)n * (n / 2) / pairs) b = (long long)n * (n / 2) / pairs;
    return (size_t)b > room ? (int)room : (int)b;
}

}  // namespace lbmgb
