// Landmark bounds: farness lower bounds that stop a lattice's sources before
// their BFS starts.
//
// On a high-diameter graph Lemma 1's bound bites only after about half the
// search (the vertices not reached yet are all taken to lie at distance
// d + 2), so BFSCut scans more than half of m n arcs.  The triangle
// inequality gives a far better bound there: with d_i(.) the distances from a
// landmark i of v's component,
//     d(v, w) >= |d_i(v) - d_i(w)|   for every i, so
//     f(v)    >= sum over w of max_i |d_i(v) - d_i(w)|,
// and, weaker but free, f(v) >= max_i sum_w |d_i(v) - d_i(w)|, which the
// sizes of landmark i's BFS levels give (the level-based bound of Bergamini,
// Borassi, Crescenzi, Marino, Meyerhenke, "Computing top-k Closeness
// Centrality Faster in Unweighted Graphs", ALENEX 2016).  A source whose
// bound ranks after the k-th key cannot enter the top-k: the same rule as
// BFSCut's, with the same ties, so the results are the same.
//
//   1. k_landmarks      four BFS by one CTA: a vertex of the largest
//                       component (of a sample), then each time the vertex
//                       farthest from the landmarks so far (on a grid:
//                       corners).  Distances, level sizes.
//   2. k_lm_bound1      the one-landmark bounds; the sources are sorted by
//                       them, so the most central ones run first (k_lattice on
//                       a few hundred) and the threshold is near its end value
//                       before the others are looked at.
//   3. k_lm_keep        sources that the one-landmark bound does not stop;
//   4. k_lm_joint       their joint bound, sums over all w (n^2 pairs of 8
//                       float operations: whole numbers below 2^24, exact) --
//                       first for a sample: where that stops under 1/16 of it
//                       (graphs whose distances concentrate) the rest is left.
//   5. k_lm_keep        again, with the joint bound; k_lattice runs what is left.
//
// Damaged grids, top-10, k_lattice alone -> with the bounds: 128^2 4.9 -> 1.6
// ms, 256^2 30.6 -> 3.4, 512^2 385 -> 14.2, 1024^2 about 12 s -> 135 ms; the
// searches visit 0.1% of n^2 vertices at 512^2 instead of 57%.  What is left
// there: the four BFS 5.5 ms (3,600 levels of about 1.5 us, a chain of one
// L2 load, two shared-memory atomics and a barrier), the joint bound 6.5 ms
// (105,000 sources: at its issue limit), the searches 2.5 ms.
#include <cuda_runtime.h>

#include "lattice.cuh"

namespace bcm {

constexpr u32 kLmQueue = 2048;      // entries of each BFS queue in shared memory
constexpr u32 kLmMaxDist = 65535;   // 256 distances up to this sum exactly in a float
constexpr u32 kLmSample = 512;
constexpr float kLmNone = -1.0f;    // dist.x of a vertex outside the landmarks' component

static size_t lm_al(size_t b) { return (b + 255) & ~(size_t)255; }

size_t landmark_bytes(uint32_t n) {
    const size_t w = lm_al(((size_t)n + 1) * 4);
    return lm_al((size_t)n * 16) + w + 4 * w + lm_al(((size_t)n + 1) * 32) + 2 * w + sparse_bitmap_bytes(n) +
           2 * lm_al((size_t)n * 8) + lm_al(kLmSample * 8) + 6 * w + lm_al(radix_scratch_bytes(n)) + 256;
}

Landmarks landmark_carve(void* base, uint32_t n) {
    char* p = (char*)base;
    auto take = [&](size_t b) { char* r = p; p += lm_al(b); return r; };
    const size_t w = lm_al(((size_t)n + 1) * 4);
    Landmarks L;
    L.dist = (float4*)take((size_t)n * 16);
    L.mind = (uint32_t*)take(w);
    L.lv_cnt = (uint32_t*)take(4 * w);
    L.lv_sum = (unsigned long long*)take(((size_t)n + 1) * 32);
    L.queue = (uint32_t*)take(2 * w);
    L.bitmap = (uint32_t*)take(sparse_bitmap_bytes(n));
    L.lb = (unsigned long long*)take((size_t)n * 8);
    L.joint = (unsigned long long*)take((size_t)n * 8);
    L.sample = (unsigned long long*)take(kLmSample * 8);
    L.key = (uint32_t*)take(w);
    L.key_tmp = (uint32_t*)take(w);
    L.val = (uint32_t*)take(w);
    L.val_tmp = (uint32_t*)take(w);
    L.list_a = (uint32_t*)take(w);
    L.list_b = (uint32_t*)take(w);
    L.radix = take(radix_scratch_bytes(n));
    L.info = (Landmarks::Info*)take(sizeof(Landmarks::Info));
    return L;
}

// Four BFS one after another by one CTA, level by level as in k_lattice
// (one barrier a level, the bitmap and the queues' fronts in shared memory).
template <int THREADS, int RW, bool SMEM>
__global__ void __launch_bounds__(THREADS) k_landmarks(GraphDev G, const u32* lat_rows, Landmarks L) {
    extern __shared__ __align__(16) u32 s_dyn[];
    __shared__ u32 s_qn[3];
    __shared__ unsigned long long s_best;
    const u32 tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const u32 n = G.n, words = (n + 31) / 32;
    u32* const bm = SMEM ? s_dyn : L.bitmap;
    u32* const sq = s_dyn + (SMEM ? sparse_bitmap_bytes(n) / sizeof(u32) : 0);
    const uint4* const rows = (const uint4*)lat_rows;
    float* const dist = (float*)L.dist;
    if (tid == 0) s_best = 0;
    __syncthreads();
    // the first landmark: of 1024 vertices spread over the ids, one of the
    // largest component, the smallest id among those
    unsigned long long best = 0;
    for (u32 i = tid; i < 1024; i += THREADS) {
        const u32 v = (u32)(((unsigned long long)i * n) >> 10);
        const unsigned long long key = ((unsigned long long)__ldg(&G.xlo[v]) << 32) | (0xffffffffu - v);
        best = key > best ? key : best;
    }
    atomicMax(&s_best, best);
    __syncthreads();
    u32 start = 0xffffffffu - (u32)s_best;
    if (tid == 0) L.info->size = (u32)(s_best >> 32);
    bool valid = true;
    for (int i = 0; i < 4 && valid; ++i) {
        __syncthreads();
        for (u32 j = tid; j < words; j += THREADS) bm[j] = 0;
        if (tid == 0) s_best = 0;
        __syncthreads();
        if (tid == 0) {
            bm[start >> 5] = 1u << (start & 31);
            sq[0] = start;
            s_qn[0] = 1;
            s_qn[1] = 0;
        }
        __syncthreads();
        u32 a = 0, b = 1, c = 2;
        u32 d = 0, reached = 0;
        u64 sum = 0;
        best = 0;
        for (;; ++d) {
            const u32 cnt = s_qn[a];
            if (cnt == 0) break;
            if (d > kLmMaxDist) { valid = false; break; }
            reached += cnt;
            sum += (u64)d * cnt;
            if (tid == 0) {
                s_qn[c] = 0;
                L.lv_cnt[(size_t)i * (n + 1) + d] = reached;
                L.lv_sum[(size_t)i * (n + 1) + d] = sum;
            }
            const u32* qc = (d & 1) ? sq + kLmQueue : sq;
            u32* qn = (d & 1) ? sq : sq + kLmQueue;
            const u32* gqc = L.queue + (size_t)(d & 1) * n;
            u32* gqn = L.queue + (size_t)((d & 1) ^ 1) * n;
            for (u32 e0 = wid * 32; e0 < cnt; e0 += THREADS) {
                const u32 e = e0 + lane;
                u32 r[RW], u = 0, near = 0;
#pragma unroll
                for (int j = 0; j < RW; ++j) r[j] = start;   // no entry: a visited vertex
                if (e < cnt) {
                    u = (e < kLmQueue ? qc[e] : __ldcg(&gqc[e])) & kLatIdMask;
                    load_row<RW>(rows, u, r);
                    near = i ? __ldcg(&L.mind[u]) : d;
                }
                u32 w[RW], found = 0;
#pragma unroll
                for (int j = 0; j < RW; ++j) {
                    const u32 k = (r[j] & kLatIdMask) >> 5;
                    w[j] = SMEM ? bm[k] : __ldcg(&bm[k]);
                }
#pragma unroll
                for (int j = 0; j < RW; ++j) {
                    const u32 k = (r[j] & kLatIdMask) >> 5;
                    const u32 seen = __funnelshift_r(w[j], 0, r[j]) & 1u;
                    const u32 old = set_if_clear<SMEM>(&bm[k], __funnelshift_l(0, 1u, r[j]), seen);
                    w[j] = ~__funnelshift_r(old, 0, r[j]) & 1u;
                    found += w[j];
                }
                u32 off, total;
                warp_places<RW>(found, off, total);
                if (total) {
                    u32 at = 0;
                    if (lane == 0) at = atomicAdd(&s_qn[b], total);
                    u32 k = __shfl_sync(0xffffffffu, at, 0) + off;
#pragma unroll
                    for (int j = 0; j < RW; ++j) {
                        if (w[j]) {
                            if (k < kLmQueue) qn[k] = r[j];
                            else gqn[k] = r[j];
                        }
                        k += w[j];
                    }
                }
                if (e < cnt) {
                    near = near < d ? near : d;
                    L.mind[u] = near;
                    dist[(size_t)u * 4 + i] = (float)d;
                    const unsigned long long key = ((unsigned long long)near << 32) | (0xffffffffu - u);
                    best = key > best ? key : best;
                }
            }
            __syncthreads();
            const u32 t = a; a = b; b = c; c = t;
        }
        if (tid == 0) L.info->levels[i] = d;
        for (int o = 16; o; o >>= 1) {
            const unsigned long long t = __shfl_xor_sync(0xffffffffu, best, o);
            best = t > best ? t : best;
        }
        if (lane == 0) atomicMax(&s_best, best);
        __syncthreads();
        start = 0xffffffffu - (u32)s_best;   // farthest from the landmarks so far
    }
    if (tid == 0) {
        L.info->valid = valid ? 1u : 0u;
        L.info->n_a = 0;
        L.info->n_b = 0;
        L.info->go = 0;
    }
}

__global__ void k_lm_clear(Landmarks L, u32 n) {
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t v = blockIdx.x * (size_t)blockDim.x + threadIdx.x; v < n; v += stride) {
        L.dist[v] = make_float4(kLmNone, kLmNone, kLmNone, kLmNone);
        L.joint[v] = 0;
    }
    if (blockIdx.x == 0)
        for (u32 i = threadIdx.x; i < kLmSample; i += blockDim.x) L.sample[i] = 0;
}

// The one-landmark bounds, and the sort keys: the top bits of the bound as a
// float (ascending with it); sources without a bound come last.
__global__ void k_lm_bound1(GraphDev G, Landmarks L, const u32* sources, u32 n_src) {
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    const u32 n = G.n, size = L.info->size;
    const bool valid = L.info->valid != 0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n_src; i += stride) {
        const u32 v = sources[i];
        const float4 t4 = L.dist[v];
        u64 lb = 0;
        u32 key = 0xffffffu;
        if (valid && t4.x != kLmNone) {
            const float t[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const u32 d = (u32)t[j];
                const size_t row = (size_t)j * (n + 1);
                const u64 c = L.lv_cnt[row + d], s = L.lv_sum[row + d], all = L.lv_sum[row + L.info->levels[j] - 1];
                const u64 b = (u64)d * c - s + (all - s) - (u64)d * (size - c);
                lb = b > lb ? b : lb;
            }
            key = __float_as_uint(__ull2float_rd(lb)) >> 7;   // below 2^24: the sign bit is 0
        }
        L.lb[v] = lb;
        L.key[i] = key;
        L.val[i] = v;
    }
}

// Sources that their bound does not stop, appended to `out` (in nearly the
// order they come in); the others are counted as cut (and as run by the
// one-source kernel, whose first test this is).
__global__ void __launch_bounds__(256) k_lm_keep(WaveParams p, Landmarks L, const u32* in, const u32* in_n, u32 first,
                                                 u32 last, bool joint, u32* out, u32* out_n) {
    __shared__ ThrCache s_thr;
    if (threadIdx.x == 0) {
        s_thr.valid = 0; s_thr.N = 0; s_thr.F = 1; s_thr.id = 0;
        read_thresholds(p.topk, s_thr);
    }
    __syncthreads();
    const u32 end = in_n ? *in_n : last;
    u32 cut = 0;
    for (size_t i0 = first + blockIdx.x * (size_t)256 + (threadIdx.x & ~31u); i0 < end; i0 += (size_t)gridDim.x * 256) {
        const size_t i = i0 + (threadIdx.x & 31);
        bool keep = false;
        u32 v = 0;
        if (i < end) {
            v = in[i];
            u64 lb = L.lb[v];
            if (joint && L.joint[v] > lb) { lb = L.joint[v]; L.lb[v] = lb; }
            keep = !bound_stops(lb, __ldg(&p.g.xlo[v]), v, s_thr);
            cut += !keep;
        }
        warp_append(keep, v, out, out_n);
    }
    cut = __reduce_add_sync(0xffffffffu, cut);
    if ((threadIdx.x & 31) == 0 && cut) {
        atomicAdd(&p.stats[ST_CUT], (unsigned long long)cut);
        atomicAdd(&p.stats[ST_WAVES], (unsigned long long)cut);
    }
}

// Joint bounds of the sources in list_a (or of kLmSample of them, spread
// evenly).  A block takes 512 sources, four per thread in registers, and a
// range of the vertices w, whose distances it stages in shared memory 256 at
// a time (one broadcast 16-byte load then serves four sources: 32 float
// operations); a float sum of 256 whole numbers up to 65535 is exact, and is
// added up in 64 bits.  The ranges are as many as give every block some work.
// Bound by issue: FADD with two operands' signs folded in and FMNMX on
// absolute values, 8 instructions a pair.
__global__ void __launch_bounds__(128) k_lm_joint(Landmarks L, u32 n, bool sample) {
    __shared__ float4 s_w[256];
    __shared__ u32 s_n;
    const u32 tid = threadIdx.x, lane = tid & 31;
    if (!L.info->valid || (!sample && !L.info->go)) return;
    const u32 na = L.info->n_a;
    const u32 ns = sample && na > kLmSample ? kLmSample : na;
    if (ns == 0) return;
    const u32 tiles = (ns + 511) / 512;
    u32 ranges = (4 * gridDim.x + tiles - 1) / tiles;
    const u32 most = (n + 1023) / 1024;
    ranges = ranges < most ? ranges : most;
    const u32 len = ((n + ranges - 1) / ranges + 255) & ~255u;
    for (u32 item = blockIdx.x; item < tiles * ranges; item += gridDim.x) {
        const u32 tile = item % tiles, w0 = (item / tiles) * len;
        const u32 w1 = w0 + len < n ? w0 + len : n;
        float4 q[4];
        u32 v[4];
        u64 sum[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const u32 i = tile * 512 + j * 128 + tid;
            v[j] = 0xffffffffu;
            q[j] = make_float4(0, 0, 0, 0);
            sum[j] = 0;
            if (i < ns) {
                v[j] = L.list_a[sample ? (u32)((u64)i * na / ns) : i];
                q[j] = L.dist[v[j]];
                if (q[j].x == kLmNone) v[j] = 0xffffffffu;   // another component: no bound
            }
        }
        for (u32 w = w0; w < w1; w += 256) {
            __syncthreads();
            if (tid == 0) s_n = 0;
            __syncthreads();
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const u32 x = w + j * 128 + tid;
                const float4 t = x < w1 ? L.dist[x] : make_float4(kLmNone, 0, 0, 0);
                const u32 m = __ballot_sync(0xffffffffu, t.x != kLmNone);
                u32 at = 0;
                if (lane == 0) at = atomicAdd(&s_n, __popc(m));
                at = __shfl_sync(0xffffffffu, at, 0);
                if (t.x != kLmNone) s_w[at + __popc(m & lanemask_lt())] = t;
            }
            __syncthreads();
            const u32 cnt = s_n;
            float acc[4] = {0, 0, 0, 0};
#pragma unroll 4
            for (u32 k = 0; k < cnt; ++k) {
                const float4 t = s_w[k];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float m = fmaxf(fmaxf(fabsf(q[j].x - t.x), fabsf(q[j].y - t.y)),
                                          fmaxf(fabsf(q[j].z - t.z), fabsf(q[j].w - t.w)));
                    acc[j] += m;
                }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) sum[j] += (u32)acc[j];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (v[j] != 0xffffffffu && sum[j])
                atomicAdd(sample ? &L.sample[tile * 512 + j * 128 + tid] : &L.joint[v[j]], (unsigned long long)sum[j]);
    }
}

// Is the joint bound worth taking?  One thread per sampled source.
__global__ void __launch_bounds__(512) k_lm_decide(WaveParams p, Landmarks L) {
    __shared__ ThrCache s_thr;
    __shared__ u32 s_cut;
    if (threadIdx.x == 0) {
        s_thr.valid = 0; s_thr.N = 0; s_thr.F = 1; s_thr.id = 0;
        read_thresholds(p.topk, s_thr);
        s_cut = 0;
    }
    __syncthreads();
    const u32 na = L.info->n_a, ns = na > kLmSample ? kLmSample : na, i = threadIdx.x;
    if (i < ns) {
        const u32 v = L.list_a[(u32)((u64)i * na / ns)];
        if (bound_stops(L.sample[i], __ldg(&p.g.xlo[v]), v, s_thr)) atomicAdd(&s_cut, 1u);
    }
    __syncthreads();
    if (i == 0) L.info->go = s_cut * 16 >= ns ? 1u : 0u;
}

// ------------------------------------------------------------- launchers
template <int T>
static int lm_launch(const WaveParams& p, const Landmarks& L, int rw, cudaStream_t s) {
    const bool smem = lattice_smem(p.g.n);
    void (*k)(GraphDev, const u32*, Landmarks) =
        rw == 4 ? (smem ? k_landmarks<T, 4, true> : k_landmarks<T, 4, false>)
                : (smem ? k_landmarks<T, 8, true> : k_landmarks<T, 8, false>);
    const size_t dyn = (smem ? sparse_bitmap_bytes(p.g.n) : 0) + 2 * kLmQueue * sizeof(u32);
    if (cudaFuncSetAttribute((const void*)k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(sparse_bitmap_bytes(kLatSmemMaxN) + 2 * kLmQueue * sizeof(u32))) != cudaSuccess)
        return -1;
    k<<<1, T, dyn, s>>>(p.g, p.lat_rows, L);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_landmarks(const WaveParams& p, const Landmarks& L, int rw, uint32_t n_src, uint32_t** order,
                     cudaStream_t s) {
    const uint32_t n = p.g.n;
    const unsigned bn = (n + 255) / 256 < 4864 ? (n + 255) / 256 : 4864;
    const unsigned bs = (n_src + 255) / 256 < 4864 ? (n_src + 255) / 256 : 4864;
    k_lm_clear<<<bn, 256, 0, s>>>(L, n);
    // about one thread per vertex of an average frontier
    if (n <= (1u << 15) ? lm_launch<128>(p, L, rw, s) : n <= (1u << 19) ? lm_launch<512>(p, L, rw, s)
                                                                         : lm_launch<1024>(p, L, rw, s))
        return -1;
    k_lm_bound1<<<bs, 256, 0, s>>>(p.g, L, p.sources, n_src);
    note_launch(3);
    bool in_tmp = false;
    if (radix_sort_pairs_u32(L.key, L.val, L.key_tmp, L.val_tmp, n_src, 24, L.radix, s, &in_tmp)) return -1;
    *order = in_tmp ? L.val_tmp : L.val;
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_landmark_filter(const WaveParams& p, const Landmarks& L, const uint32_t* order, uint32_t first,
                           uint32_t n_src, cudaStream_t s) {
    const unsigned b = (n_src + 255) / 256 < 1216 ? (n_src + 255) / 256 : 1216;
    k_lm_keep<<<b, 256, 0, s>>>(p, L, order, nullptr, first, n_src, false, L.list_a, &L.info->n_a);
    k_lm_joint<<<152 * 8, 128, 0, s>>>(L, p.g.n, true);
    k_lm_decide<<<1, 512, 0, s>>>(p, L);
    k_lm_joint<<<152 * 8, 128, 0, s>>>(L, p.g.n, false);
    k_lm_keep<<<b, 256, 0, s>>>(p, L, L.list_a, &L.info->n_a, 0, 0, true, L.list_b, &L.info->n_b);
    note_launch(5);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace bcm
