// Rows into which the standalone adjoint deals the 32-tile chunks of every
// super cell (plain C++: a host rule).
#pragma once

#include <stdint.h>

namespace serbf {

// One row per chunk of the fullest super cell (most), so that a warp never
// takes two chunks of a super cell in turn, but at most four times the average
// super cell's chunks and four more, or what the warps' lanes cover in a few
// passes (kRowPasses in backward.cu): a kernel's warps look at every row of
// every super cell in its support, and one dense super cell must not make them
// look at that many empty rows in all the others.  With half of 400 000 points
// in one super cell (196 chunks) and 512 kernels the adjoint took 1030 us by
// whole super cells, 590 with a row per chunk, now 315; half of 10^6 points (488
// chunks), 300 kernels: 3300, 2250 and 660.
inline int chunk_rows(int64_t tiles, int64_t supers, int most) {
    const int64_t fair = 4 * (tiles / (32 * (supers > 0 ? supers : 1))) + 4;
    return (int)(most < fair ? most : fair);
}

}  // namespace serbf
