// sort_plan.cuh -- how many keys a thread of the radix sort takes and how many
// blocks a sort may need. Used by the kernel (which knows the key count) and by
// the host (which sizes grid and look-back words for the capacity).
#pragma once

#include <algorithm>
#include <cstdint>

#ifdef __CUDACC__
#define GI_HOST_DEVICE __host__ __device__
#else
#define GI_HOST_DEVICE
#endif

namespace gi {

constexpr int kSortThreads = 512;   // threads per onesweep block
constexpr int kSortMaxItems = 16;   // keys per thread at most

// Keys per thread for K keys; wave = blocks that run at the same time (one per
// SM). A block is latency-bound (ranking key by key, barriers, look-back) and
// fills an SM's registers, so the sort takes as long as its waves: the fewest
// keys a thread that need one wave, beyond that 12 if that needs no more waves
// than 16. Measured on 152 SMs with 512 threads at 16 / 12 / 8 / 4 keys (256 x
// 16 before): render of 1,000 x 1,422 / 51,000 Gaussians 67 / - / 59 / 56 us
// (65), 2040x1356 / 100,000 85 / - / 79.5 / 80.4 (90.7), 1,738 x 1,506 / 130,000
// 98 / 94.5 / 101 / 101 (104), 1,827 x 1,396 / 200,000 124 / - / 130 / 132 (130);
// step of 1,633 x 1,443 / 104,000 at tile 8 316 / 310.5; 24 keys gain 5 us more
// there and cost 1 us everywhere else (spills).
GI_HOST_DEVICE inline int sort_items(int K, int wave) {
    const int w = wave * kSortThreads;  // keys of one wave per item
    if (K <= 4 * w) return 4;
    if (K <= 8 * w) return 8;
    int k12 = 12 * w, k16 = 16 * w;  // keys of the waves that 16 keys a thread take
    while (K > k16) {                // (two divisions instead: 0.2 us a pass)
        k12 += 12 * w;
        k16 += 16 * w;
    }
    return K <= k12 ? 12 : 16;
}

// Blocks that a sort of up to `capacity` keys may use (sort_items: never more
// than the waves that 16 keys a thread take).
inline int64_t sort_blocks(int64_t capacity, int wave) {
    const int64_t by4 = (capacity + kSortThreads * 4 - 1) / (kSortThreads * 4);
    const int64_t wave16 = int64_t(wave) * kSortThreads * kSortMaxItems;
    return std::max<int64_t>(1, std::min<int64_t>(by4, wave * ((capacity + wave16 - 1) / wave16)));
}

}  // namespace gi
