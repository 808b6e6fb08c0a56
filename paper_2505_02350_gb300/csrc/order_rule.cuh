// When one launch makes the forward's heavy-first item order (plain C++: a host
// rule, restated by Problem.launches_per_epoch).
#pragma once

#include <stdint.h>

namespace serbf {

constexpr int64_t kOrderDirectItems = 1 << 16;

// Up to so many items, counted as the most that a field can have (one per 64
// points and one per super cell with points), so that the rule needs nothing
// that only the device knows.  Rebuild with the order in one launch / in two, us:
// 32^3 points 29 / 33, 128^3 (32 768 items) 32 / 35, 160^3 (64 000) 29 / 33, but
// 300 000 points in 97 336 super cells (93 000 items) 231 / 225: every block
// counts all classes.
inline bool order_direct(int64_t points, int64_t supers) {
    return points / 64 + (supers < points ? supers : points) <= kOrderDirectItems;
}

}  // namespace serbf
