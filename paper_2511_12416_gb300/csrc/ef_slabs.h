// How a Raw Estimate call runs over its slabs of items, apart from CUDA: the
// order of launches and joins of the two streams.
#pragma once

#include <stdint.h>

#include <algorithm>

namespace ef {

// Images (one per bitstring) that a slab of `slab` items may touch: a slab need not
// begin or end with a bitstring's first or last chunk.
inline int64_t slab_images(int64_t nb, int64_t slab, int64_t n_chunks) {
    return std::min<int64_t>(std::max<int64_t>(nb, 1), slab / n_chunks + 2);
}

// (bitstring, chunk) items per slab: as many as `budget` bytes hold, whole
// bitstrings where one fits. item, image: bytes of an item's samples and of a
// bitstring's image; blocks: Philox blocks of the call. (The images at a slab's
// ends count, so that a slab stays within the budget.)
// Several slabs in flight are worth it from about two waves of the evaluation's
// CTAs each and some milliseconds of sampling (10^9 Philox blocks): then a call is
// cut in four even where fewer slabs would hold it.
inline int64_t slab_items_of(int64_t nb, int64_t n_chunks, int64_t n_seg, int64_t item, int64_t image, int64_t budget, int64_t sms,
                             double blocks) {
    const int64_t items = std::max<int64_t>(nb, 1) * n_chunks;
    const int64_t bytes = image + item * n_chunks;  // of a whole bitstring
    const int64_t room = budget - 2 * image;
    const bool whole = bytes <= room;
    int64_t slab = whole ? std::min<int64_t>(room / bytes, 1 << 20) * n_chunks
                         : std::max<int64_t>(1, room / std::max<int64_t>(item, 1));
    slab = std::min(std::min(slab, items), std::max<int64_t>(1, 2147483647ll / n_seg));
    const int64_t wave = 2 * sms, quarter = (items + 3) / 4;
    if (whole && items >= 4 * wave && slab > quarter && blocks >= 1e9)
        slab = std::min(slab, (std::max<int64_t>(2 * wave, quarter) + n_chunks - 1) / n_chunks * n_chunks);
    return slab;
}

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
