// Tiles of the radix sort (lbvh.cu); plain C++, so that the sizes can be checked
// without a GPU.
#pragma once

#include <cstdint>
#include <type_traits>

namespace meshgs {

constexpr int kSortTileMin = 1024;    // keys per sort tile: 1024, 2048, 4096 or 8192
// Tiles whose counts a pass sums itself, in every block: 2M keys (245 tiles) take 214 us
// so; 2.3M (281) 224, and 198 when k_sort_scan sums them; 4M (489) 477 and 341.
constexpr int kSortTilesMax = 256;

// Threads and keys per thread of a sort of n keys: f gets them as compile-time
// constants.  Tiles grow with n: a pass reads every tile's 256 counts in every
// block, 1 KB x tiles^2 in all, against 8 B x n of keys -- at most about 250 tiles
// up to 2M keys.  Smaller tiles than these spread the ranking over more SMs.
template <typename F> inline void sort_shape(int n, F f) {
    using std::integral_constant;
    if (n <= 160 * 1024) f(integral_constant<int, 256>(), integral_constant<int, 4>());
    else if (n <= 480 * 1024) f(integral_constant<int, 256>(), integral_constant<int, 8>());
    else if (n <= 1024 * 1024) f(integral_constant<int, 512>(), integral_constant<int, 8>());
    else f(integral_constant<int, 512>(), integral_constant<int, 16>());
}

// Tiles of n keys (any int: n + a tile would overflow at the top of the range).
inline int sort_tiles(int n) {
    int T = 0;
    sort_shape(n, [&](auto th, auto it) {
        const int64_t tile = th.value * it.value;
        T = (int)((n + tile - 1) / tile);
    });
    return T;
}

}  // namespace meshgs
