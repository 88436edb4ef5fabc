// How many entries the randomized PROBE's level lists are sized for.  Plain host code: the host sizes the list that a
// level writes by rand_list_entries, and tells the level how much work it may do by rand_list_items, which is defined by
// the former, so that a list sized for a level always takes that level.  (With two roundings of the share, one to size
// and one to accept, a list kept from an earlier call could be large enough by the one and too small by the other.)
#pragma once

#include <algorithm>
#include <cstdint>

namespace ps {

constexpr int64_t kRandListMin = 1024;  // entries; below it the share of the items says little

// Entries that a level of E work items is sized for: `share` (0 < share <= 1) of them, at least kRandListMin, and never
// more than one an item (an item finds at most one member).  Grows with E.
inline int64_t rand_list_entries(double share, int64_t E) {
    return std::min<int64_t>(E, std::max<int64_t>(kRandListMin, (int64_t)(share * (double)E) + 1));
}

// The most work items whose level a list of `cap` entries is sized for: the largest E with rand_list_entries(share, E)
// <= cap.
inline int64_t rand_list_items(double share, int64_t cap) {
    if (cap < kRandListMin) return std::max<int64_t>(0, cap);
    int64_t E = (int64_t)((double)cap / share) + 2;  // at least the answer; one entry is 1 / share items
    while (rand_list_entries(share, E) > cap) --E;
    return E;
}

}  // namespace ps
