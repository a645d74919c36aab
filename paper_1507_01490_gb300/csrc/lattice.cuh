// What the kernels on padded rows share (lattice.cu, landmark.cu).
#pragma once
#include "internal.h"

namespace bcm {

constexpr u32 kLatSmemMaxN = 1600000;    // bitmap in shared memory up to this n (200 KB)
constexpr u32 kLatIdMask = 0x0fffffffu;  // neighbour id; the degree is above it

// Sets `bit` of a bitmap word where `seen` says that it was clear, and
// returns the word as it was (all ones where nothing was done): predicated
// by hand, since the compiler branches around each of a row's atomics.
template <bool SMEM>
__device__ __forceinline__ u32 set_if_clear(u32* word, u32 bit, u32 seen) {
    u32 old = ~0u;
    if (SMEM) {
        const u32 at = (u32)__cvta_generic_to_shared(word);
        asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.u32 p, %3, 0;\n\t@p atom.shared.or.b32 %0, [%1], %2;\n\t}"
                     : "+r"(old) : "r"(at), "r"(bit), "r"(seen) : "memory");
    } else {
        asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.u32 p, %3, 0;\n\t@p atom.global.or.b32 %0, [%1], %2;\n\t}"
                     : "+r"(old) : "l"(__cvta_generic_to_global(word)), "r"(bit), "r"(seen) : "memory");
    }
    return old;
}

// Row of vertex u: RW entries.
template <int RW>
__device__ __forceinline__ void load_row(const uint4* rows, u32 u, u32 (&r)[RW]) {
#pragma unroll
    for (int j = 0; j < RW; j += 4) {
        const uint4 t = __ldg(&rows[(size_t)u * (RW / 4) + j / 4]);
        r[j] = t.x; r[j + 1] = t.y; r[j + 2] = t.z; r[j + 3] = t.w;
    }
}

// A thread's place in a list to which every thread of the warp appends `found`
// entries (at most RW): the entries before its own, and the warp's total; a
// scan of the counts, bit by bit.
template <int RW>
__device__ __forceinline__ void warp_places(u32 found, u32& off, u32& total) {
    const u32 lt = lanemask_lt();
    off = 0;
    total = 0;
#pragma unroll
    for (int k = 0; (1 << k) <= RW; ++k) {
        const u32 m = __ballot_sync(0xffffffffu, (found >> k) & 1u);
        off += __popc(m & lt) << k;
        total += __popc(m) << k;
    }
}

}  // namespace bcm
