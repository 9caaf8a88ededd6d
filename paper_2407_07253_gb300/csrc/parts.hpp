// Work lists that share a bounded scratch, launched part by part.
#pragma once
#include <algorithm>
#include <vector>

// Splits consecutive items of the given sizes into parts of at most cap in all
// (an item larger than cap is a part of its own): off[i] is item i's place within
// its part, part k holds the items first[k] .. first[k + 1] - 1.  Returns the
// largest part's size.
inline long long split_parts(const std::vector<long long>& size, long long cap, std::vector<long long>& off,
                             std::vector<int>& first) {
    off.clear();
    first.assign(1, 0);
    long long used = 0, most = 0;
    for (size_t i = 0; i < size.size(); ++i) {
        if (used > 0 && used + size[i] > cap) {
            first.push_back((int)i);
            used = 0;
        }
        off.push_back(used);
        used += size[i];
        most = std::max(most, used);
    }
    if (!size.empty()) first.push_back((int)size.size());
    return most;
}
