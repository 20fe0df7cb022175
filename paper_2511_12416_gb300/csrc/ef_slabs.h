// How a Raw Estimate call runs over its slabs of items, apart from CUDA: the
// order of launches and joins of the two streams.
#pragma once

#include <stdint.h>

#include <algorithm>

namespace ef {

// Trajectories of a (bitstring, chunk) item: a multiple of 128, at most 2^25. Enough
// items for about four waves of three CTAs per SM, one chunk per bitstring where
// the bitstrings alone give them. segment, seg_bytes: trajectories of a segment's
// four streams and bytes of their samples (0: none are kept).
// A slab of fewer items than two waves of two CTAs per SM is all tail: where many
// flips make long items larger than that, they are cut so that a slab holds 12 per SM.
// 64 uneven circuits, 10^5 and more trajectories for each of many bitstrings: 42.3 s
// uncut, 34.9 s at 6 per SM, 33.7 s at 12, 33.8 s at 24. Cutting the 52-qubit LUCJ
// circuit's items too, whose slabs hold 800, costs 4-6 % (6-12 per SM). Every item has
// 88 bytes of partial sums for the whole call, so no cut makes more than 2^24 of them
// unless an item would not fit half a slab.
inline int64_t chunk_trajectories(int64_t nb, int64_t t, int64_t sms, int64_t segment, int64_t seg_bytes, int64_t slab_bytes) {
    const auto ceil_div = [](int64_t a, int64_t b) { return (a + b - 1) / b; };
    const auto up128 = [&](int64_t x) { return ceil_div(x, 128) * 128; };
    const int64_t target = sms * 3 * 4, bits = std::max<int64_t>(nb, 1);
    const int64_t chunks = std::min(std::max<int64_t>(1, ceil_div(target, bits)), std::max<int64_t>(1, t / 256));
    const int64_t per = std::min<int64_t>(up128(ceil_div(t, chunks)), (int64_t)1 << 25);
    if (seg_bytes == 0 || ceil_div(per, segment) * seg_bytes <= slab_bytes / (4 * sms)) return per;
    const int64_t most = std::max<int64_t>(1, slab_bytes / target / seg_bytes) * segment;
    const int64_t half = std::max<int64_t>(1, slab_bytes / 2 / seg_bytes) * segment;  // a slab holds an item whatever its length
    const int64_t parts = std::min(ceil_div(t, most), ((int64_t)1 << 24) / bits);
    return up128(ceil_div(t, std::max(parts, ceil_div(t, std::min(per, half)))));
}

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
