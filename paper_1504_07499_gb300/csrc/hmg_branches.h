// How many RVEs the engine advances at once (host only).
#pragma once

#include <stddef.h>

namespace hmg {

// RVEs advanced at once within a tick (branches of the engine's graph), for `live` unfinished
// entries whose FP32 fields and spectra take `bytes` together: as many entries of the mean size
// as keep these within half of the L2 through a block of four sweeps, 3 to 16.  Small grids need
// many to fill the GPU (an x pass of one RVE is 18 CTAs at 16^3), large ones evict each
// other.  ms per batch at 2, 3, 4, 6, 8, 16 branches:
//   48 x 16^3  74.3 56.9 49.5 40.3 35.9 28.9     24 x 24^3  42.6 32.6 28.0 23.2 20.8 19.9
//   24 x 32^3  52.2 40.8 36.1 30.8 29.1 29.1     12 x 48^3  37.4 32.9 32.1 31.7 31.9 32.1
//   12 x 64^3  40.9 38.5 38.5 39.2 39.8 44.2     8 x 96^3   81.5 88.1 94.2 91.1 94.4 94.5
//   6 x 128^3  133 132 132 131 131 132           5 x 64^3 + 4 x 96^3 + 3 x 128^3  127 126 130 133 135 143
inline size_t side_branches(size_t live, size_t bytes) {
    if (live == 0 || bytes == 0) return 3;
    const size_t fit = (64u << 20) / (bytes / live);
    return fit < 3 ? 3 : fit > 16 ? 16 : fit;
}

}  // namespace hmg
