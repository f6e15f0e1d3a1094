// How much memory a search asks for at once. Plain functions, so that the host
// tests run the same code.
#pragma once

#include <stdint.h>

namespace sindi {

// The largest of n, ceil(n / 2), ceil(n / 4), ... 1 for which get(size) succeeds; 0 if none does.
template <typename Get>
int64_t largest_that_fits(int64_t n, Get&& get) {
    for (; n >= 1; n = (n + 1) / 2) {
        if (get(n)) return n;
        if (n == 1) break;
    }
    return 0;
}

}  // namespace sindi
