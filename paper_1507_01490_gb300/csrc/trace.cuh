// Trace records of the BFS kernels (BCM_TRACE, BCM_TRACE_LANES; layout in
// include/bcm.h, bcm_trace).
#pragma once
#include "internal.h"

namespace bcm {

// One trace record (4 words), when tracing is on.  The second word holds
// the kind in bits 60..63, an identifier (wave or CTA) in bits 32..59 and a
// level in bits 0..31.
__device__ __forceinline__ void trace_record(const WaveParams& p, u32 kind, u32 id, u32 level, u64 a, u64 b,
                                             u64 t) {
    if (!p.trace) return;
    const u32 i = atomicAdd(p.trace_n, 1u);
    if (i >= p.trace_cap) return;
    unsigned long long* r = p.trace + 4 * (size_t)i;
    r[0] = t;
    r[1] = ((u64)kind << 60) | ((u64)(id & 0xfffffffu) << 32) | level;
    r[2] = a;
    r[3] = b;
}

// Lane records (BCM_TRACE_LANES): source v's Table 1 state before the
// stopping rule at level d, and how its BFS ended.
static __device__ __noinline__ void lane_level(const WaveParams& p, u32 v, u32 d, u64 f, u32 nd, u32 gt) {
    trace_record(p, TR_LANE_LEVEL, v, d, f, (u64)nd | ((u64)gt << 32), global_ns());
}
static __device__ __noinline__ void lane_end(const WaveParams& p, u32 v, u32 d, u64 f, u32 nd, bool cut) {
    trace_record(p, TR_LANE_END, v, d, f, (u64)nd | ((u64)(cut ? 1u : 0u) << 32), global_ns());
}

}  // namespace bcm
