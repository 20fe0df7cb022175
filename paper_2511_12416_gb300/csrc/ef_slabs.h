// How a Raw Estimate call runs over its slabs of items, apart from CUDA: the
// order of launches and joins of the two streams.
#pragma once

#include <stdint.h>

#include <algorithm>

namespace ef {

// launch(first item, items, turn) per slab; with `two`, turns 0 and 1 take the
// caller's stream and a side stream that fork() makes wait for the caller's.
// Whatever fails, join() makes the caller's stream wait for the side stream, so
// that work launched on it has ended where the caller believes the call's has.
// E: a status whose zero is success; the first failure is returned.
template <typename E, typename Fork, typename Join, typename Launch>
E for_slabs(int64_t items, int64_t slab, bool two, Fork fork, Join join, Launch launch) {
    E e{};
    if (two) {
        e = fork();
        if (e != E{}) return e;
    }
    int turn = 0;
    for (int64_t i0 = 0; i0 < items && e == E{}; i0 += slab, turn ^= two ? 1 : 0)
        e = launch(i0, std::min(slab, items - i0), turn);
    if (two) {
        const E j = join();
        if (e == E{}) e = j;
    }
    return e;
}

}  // namespace ef
