// Warps per forward work item, chosen by the number of items (plain C++: a host
// rule).
#pragma once

#include <stdint.h>

namespace serbf {

// For a field (or a batch) of items4 items of up to four tiles, unless fixed (1,
// 2, 4 or 8) says so.  Items differ in cost (an item in the middle of the kernels
// whose points all carry residuals costs five times the mean and more), so a
// launch with few items per warp waits for its heaviest ones; more warps per item
// shorten that tail and cost issue slots for barriers and short batches.  One warp
// takes items of four tiles, several take items of two: full super cells have
// twice as many of those, super cells of a tile or less as many, and both kinds
// cross at about the same number of four-tile items (by two-tile items sparse
// super cells got too many warps: 200 000 points in 15 625 of them 78 us for the
// forward instead of 62).  Measured on a 152-SM part in each split's own measured
// order, items4 and us of the fused call with 1 / 2 / 4 warps.  Full super cells:
// 256 (32^3) 36 / 35 / 35, 2.3 k (64^3 + 32^3) 104 / 59 / 61, 4 k (80^3) 133 / 82 /
// 89 (in natural order 194 / 111 / 96), 7.2 k (97^3) 129 / 124 / 135 (natural 194 /
// 140 / 141), with 4096 kernels 163 / 148 / 159 (compensated 248 / 193 / 201, but
// in natural order two are a tenth slower than four), 9 k (105^3) 145 / 137 / 164
// (natural 210 / 158 / 166), 13.5 k (120^3) 275 / 251 / 297, 16 k (128^3) 337 / 309
// / 365, 22 k (140^3) 384 / 385 / 458, 26 k (150^3) 467 / 476 / 568, 32 k 548 / 574
// / 688, 63 k 963 / 1062 / 1270, 74 k (9.4 M points of a band) 1671 / 1817 / 2109; a
// batch of 16 fields, 41 k in all, 552 / 718 / 979 an epoch.  One tile or less per
// super cell (in brackets the forward alone): 8 k 55 / 52 / 62 (37 / 40 / 47),
// 15.6 k 90 / 96 / 117 (54 / 62 / 78), 30 k 134 / 147 / 189 (88 / 102 / 131), 39 k
// 166 / 186 / 241 (111 / 128 / 166).  8 warps are within 8 % of 4 up to 256 items
// and slower above.
inline int forward_warps(int64_t items4, int sm_count, int fixed) {
    if (fixed == 1 || fixed == 2 || fixed == 4 || fixed == 8) return fixed;
    const int64_t resident = 20 * (int64_t)sm_count;  // warps in flight
    return items4 >= 8 * resident ? 1 : (2 * items4 >= 5 * resident ? 2 : 4);
}

}  // namespace serbf
