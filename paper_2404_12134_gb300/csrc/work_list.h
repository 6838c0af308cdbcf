// Sizes of a work list.  Plain C++ for host code and its tests.
#pragma once

#include <cstdint>

namespace wts {

// Whether P pairs of nb items each (a grouped list, whose last items of a
// shorter pair are empty) may be taken by int cursors: every warp takes one item
// past the list's end before it leaves, so the list and the warps stay in 31 bits.
inline bool grouped_list_fits(int64_t P, int64_t nb, int64_t warps)
{
    return P * nb + warps < ((int64_t)1 << 31);
}

}  // namespace wts
