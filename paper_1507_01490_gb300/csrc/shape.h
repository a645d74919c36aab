// Sizes and choices of the all-pairs kernel that the host makes: plain C++, so
// that they can be checked without a GPU.
#pragma once
#include <cstddef>
#include <cstdint>
#include <initializer_list>

#ifdef __CUDACC__
#define BCM_HD __host__ __device__
#else
#define BCM_HD
#endif

namespace bcm {

BCM_HD constexpr size_t al256(size_t b) { return (b + 255) & ~(size_t)255; }

// One cluster's planes: vis, two of frontiers, and each row's counts.
constexpr size_t allpairs_slot_bytes(uint32_t n, int W) { return al256((size_t)n * W * 24 + (size_t)n * 8); }

// Lanes, cluster size and cluster count for n vertices on `sms` SMs, at most
// `budget` bytes of slots; returns the SMs it keeps busy.  Where every wave of
// 64 targets has an SM of its own: that (a cluster's barrier and its loads
// past L1 cost more than idle SMs: Chung-Lu 1000 and 4000, C = 1: 0.043 and
// 0.11 ms, C = 8: 0.09 and 0.18).  Else the choice that keeps most SMs busy, of
// those the widest lanes (an arc's word then serves more targets: R-MAT 2^16,
// 256 lanes 12.2 ms, 128 13.9), of those the smallest clusters.
inline int allpairs_shape(uint32_t n, int sms, size_t budget, int lanes, int* W, int* C, int* clusters) {
    *W = *C = *clusters = 0;
    int best = 0;
    const uint32_t one = (n + 63) / 64;
    if (!lanes && one <= (uint32_t)sms && one * allpairs_slot_bytes(n, 1) <= budget) {
        *W = *C = 1;
        *clusters = (int)one;
        return (int)one;
    }
    for (int w : {4, 2, 1}) {
        if (lanes && lanes != 64 * w) continue;
        const uint32_t waves = (n + 64 * w - 1) / (64 * w);
        for (int c : {1, 2, 4, 8}) {
            size_t k = budget / allpairs_slot_bytes(n, w);
            if (k > (size_t)(sms / c)) k = (size_t)(sms / c);
            if (k > waves) k = waves;
            if ((int)k * c > best) {
                best = (int)k * c;
                *W = w;
                *C = c;
                *clusters = (int)k;
            }
        }
    }
    return best;
}

// A number coprime to `count`, near the golden ratio of it: i * step mod count, i
// = 0, 1, ..., visits every number once, and any first few are spread evenly.
inline uint32_t spread_step(uint32_t count) {
    for (uint32_t s = (uint32_t)((uint64_t)count * 618 / 1000);; ++s) {
        uint32_t a = count, b = s;
        while (b) { const uint32_t t = a % b; a = b; b = t; }
        if (a == 1) return s;
    }
}

// Is that shape worth taking?  A large graph whose planes leave L2 (`budget`)
// with most SMs idle stays on the kernels that search from sources; so does one
// that no shape fits.  With 130 MB on 152 SMs the line lies at about 284,000
// vertices.  Farness of every vertex, grid-wide kernel -> all pairs: Chung-Lu of
// 100,000 vertices and 16 arcs each 307 -> 43 ms, 200,000 687 -> 293, 283,000
// 987 -> 412, R-MAT 2^18 and 12 arcs 563 -> 455; deep graphs too (a grid-wide
// level costs two barriers of the whole grid for 128 sources): a directed path of
// 8,000 4,164 -> 43, paths of 30 in 280,000 1,020 -> 607, a ring of 131,072 and 40
// arcs 279 -> 217 s.
inline bool allpairs_fits(uint32_t n, int sms, size_t budget, int lanes, int* W, int* C, int* clusters) {
    const int busy = allpairs_shape(n, sms, budget, lanes, W, C, clusters);
    if (busy <= 0) return false;
    return busy * 4 >= sms * 3 || (uint64_t)*clusters == ((uint64_t)n + 64 * *W - 1) / (64 * *W);
}

}  // namespace bcm
