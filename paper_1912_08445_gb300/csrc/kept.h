// Buffers kept from one use to the next.
#pragma once
#include <algorithm>
#include <cstdint>

namespace mg {

// Makes room for `count` elements in a kept buffer that holds `cap` (0: there is none). It stays
// when it is large enough and not more than half empty. Otherwise alloc(n), which gives the
// old one back first and returns 0 on success, is asked for 3 % to spare for the next use, then
// for `count` itself. `cap` is what was allocated in the end.
template <class Alloc>
int kept_buffer(int64_t &cap, int64_t count, Alloc alloc) {
    if (cap > 0 && cap >= count && cap <= 2 * count + 4096) return 0;
    cap = 0;
    int64_t got = count + count / 32;
    int rc = alloc(got);
    if (rc && got > count) {
        got = count;
        rc = alloc(got);
    }
    if (!rc) cap = std::max<int64_t>(1, got);
    return rc;
}

}  // namespace mg
