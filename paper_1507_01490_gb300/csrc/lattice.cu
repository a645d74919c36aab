// BFSCut on graphs whose degrees are at most 8 (lattices, meshes, road-like
// graphs): one source per CTA, as k_sparse runs it, on a padded adjacency.
//
// k_sparse lays the arc ranges of 32 queue entries end to end and finds each
// arc's owner by a search over prefix sums: about 230 thread instructions per
// arc, two block barriers and a serial 128-bit test per level.  On a graph
// whose rows have at most 4 (or 8) arcs none of that is needed:
//
//   * the rows are copied once per graph into a padded table of 4 (or 8)
//     32-bit entries, each the neighbour's id with its degree in the top four
//     bits, so a thread takes one frontier vertex, reads its row with one (or
//     two) 16-byte loads, and knows every neighbour's degree without asking;
//   * the visited bitmap lies in shared memory where it fits (n <= 1.6 M:
//     200 KB), so a test or a set costs no trip to L2; the queues' first
//     kLatQueue entries do too, longer frontiers go on in global memory;
//   * gamma_{d+1} is the next queue's length, and every thread updates
//     (n_d, f_d) and applies the stopping rule by itself, in 64 bits: the
//     rule f~ N_k > F_k (x-1)^2 (or >=, where a tie loses on the id) is
//     f~ >= a whole number that changes only with the threshold, found once
//     by a 128-bit division by the one thread that reads the threshold.  So
//     a level has one block barrier and no serial part.
//
// What bounds it: instruction issue (60% of slots on the 256^2 grid, 13 warp
// instructions per vertex) and the barrier of short levels.  Damaged grids,
// top-10, k_sparse -> this kernel: 128^2 13.8 -> 4.4 ms, 256^2 125.6 -> 30
// ms, 512^2 1,534 -> 389 ms, 1/16 of 1024^2's sources 1.47 s -> 0.73 s.
#include <cuda_runtime.h>

#include "lattice.cuh"
#include "trace.cuh"

namespace bcm {

constexpr u32 kLatQueue = 1024;          // queue entries in shared memory, per queue
// Threads an SM holds at once (the register budget): 48 registers for rows of
// 4.  512^2: 389 ms; 1536 threads (40 registers, spills) 439, 1024 400.
constexpr int kLatResident = 1280;

bool lattice_smem(uint32_t n) { return n <= kLatSmemMaxN; }

size_t lattice_slot_bytes(uint32_t n, uint32_t qcap) {
    return (lattice_smem(n) ? 0 : sparse_bitmap_bytes(n)) + 2 * al256((size_t)qcap * sizeof(uint32_t));
}

static size_t lattice_dyn_smem(uint32_t n) {
    return (lattice_smem(n) ? sparse_bitmap_bytes(n) : 0) + 2 * kLatQueue * sizeof(u32);
}

template <int RW>
__global__ void k_lattice_rows(const u32* rp, const u32* col, u32 n, u32* rows) {
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t v = blockIdx.x * (size_t)blockDim.x + threadIdx.x; v < n; v += stride) {
        const u32 b = rp[v], e = rp[v + 1];
#pragma unroll
        for (int j = 0; j < RW; ++j) {
            u32 w = (u32)v;   // padding: the vertex itself, visited whenever its row is read
            if (b + j < e) {
                const u32 x = col[b + j];
                w = x | ((rp[x + 1] - rp[x]) << 28);
            }
            rows[v * RW + j] = w;
        }
    }
}

int launch_lattice_rows(const uint32_t* rp, const uint32_t* col, uint32_t n, int rw, uint32_t* rows, cudaStream_t s) {
    const unsigned blocks = (n + 255) / 256 < 4864 ? (n + 255) / 256 : 4864;
    if (rw == 4) k_lattice_rows<4><<<blocks, 256, 0, s>>>(rp, col, n, rows);
    else k_lattice_rows<8><<<blocks, 256, 0, s>>>(rp, col, n, rows);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// The smallest f~ that stops source v of reach x under threshold t: f~ N > F
// (x-1)^2, or >= where v loses the tie on its id.  (f~ <= n^2 < 2^60.)
__device__ __noinline__ long long cut_limit(const ThrCache& t, u32 x, u32 v) {
    const long long never = 0x7fffffffffffffffll;
    if (!t.valid || t.N == 0) return never;   // N = 0: only x = 1 could stop, and such a source has no arc
    const unsigned __int128 xm1 = x - 1;
    const unsigned __int128 rhs = (unsigned __int128)t.F * xm1 * xm1;
    const unsigned __int128 q = rhs / t.N;
    const bool even = q * t.N == rhs;
    const unsigned __int128 lim = q + ((even && v > t.id) ? 0 : 1);
    return lim > (unsigned __int128)never ? never : (long long)lim;
}

// A completed source of a top-k run: into the shared top-k unless the
// threshold ranks before it.  While another CTA holds the lock the threshold is
// read again: it only rises, and most waiters then have nothing to insert
// (before a threshold exists, thousands of sources complete together).
__device__ __noinline__ void lattice_complete(const WaveParams& p, ThrCache& t, u32 v, u64 f, u32 r) {
    u64 N, F;
    score_key(f, r, N, F);
    const u64 t0 = global_ns();
    u32 ns = 32;
    for (;;) {
        if (t.valid && ranks_before(t.N, t.F, t.id, N, F, v)) return;   // (equal: an offered key that is its own)
        if (atomicCAS(p.topk.lock, 0u, 1u) == 0u) break;
        if (global_ns() - t0 > p.lock_limit_ns) { atomicOr(p.err, DEV_ERR_LOCK_TIMEOUT); return; }
        __nanosleep(ns);
        if (ns < 1024) ns <<= 1;
        read_thresholds(p.topk, t);
    }
    __threadfence();
    topk_insert_locked(p.topk, v, f, r);
    topk_publish_locked(p.topk);
    lock_release(p.topk.lock);
}

template <int THREADS, int RW, bool SMEM>
__global__ void __launch_bounds__(THREADS, (RW == 4 ? kLatResident : 1024) / THREADS) k_lattice(WaveParams p) {
    extern __shared__ __align__(16) u32 s_dyn[];
    __shared__ u32 s_qn[3], s_ds[3];     // per level, rotating: queue length; its vertices' degree sum
    __shared__ long long s_cut[2];       // per level parity: the f~ that stops the source
    __shared__ u32 s_base, s_stop, s_skip, s_lo, s_hi;
    __shared__ unsigned long long s_st[ST_COUNT];   // ctl's counters
    __shared__ ThrCache s_thr;                      // ctl's last snapshot of the threshold
    const u32 tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const bool ctl = tid == THREADS - 32;   // reads the threshold, keeps the counters
    const GraphDev& G = p.g;
    const u32 foot = p.footnote;
    const u32 n_end = p.n_end_dev ? vload(p.n_end_dev) : p.n_end;
    const u32 words = (G.n + 31) / 32;
    char* slot = p.slot_base + (size_t)blockIdx.x * p.slot_stride;
    u32* const bm = SMEM ? s_dyn : (u32*)slot;
    u32* const sq = s_dyn + (SMEM ? sparse_bitmap_bytes(G.n) / sizeof(u32) : 0);
    u32* const gq = (u32*)(slot + (SMEM ? 0 : sparse_bitmap_bytes(G.n)));
    const u32 gstride = (u32)(al256((size_t)p.sparse_qcap * sizeof(u32)) / sizeof(u32));
    const uint4* const rows = (const uint4*)p.lat_rows;
    const bool cuts = !p.exhaustive && !p.nocut;

    if (ctl) {
        for (int i = 0; i < ST_COUNT; ++i) s_st[i] = 0;
        s_thr.valid = 0; s_thr.N = 0; s_thr.F = 1; s_thr.id = 0;
    }
    if (SMEM)
        for (u32 i = tid; i < words; i += THREADS) bm[i] = 0;

    for (;;) {
        if (tid == 0) {
            s_base = atomicAdd(p.head, 1u);
            s_stop = (s_base >= n_end) || (vload(p.err) != 0);
        }
        __syncthreads();
        if (s_stop) break;
        const u32 v = __ldg(&p.sources[s_base]);
        const u32 deg = __ldg(&G.rp[v + 1]) - __ldg(&G.rp[v]);
        const u32 x = __ldg(&G.xlo[v]);
        u64 seq = 0, eseq = 0;
        if (ctl) {
            s_st[ST_WAVES]++;
            long long lim = 0x7fffffffffffffffll;
            if (!p.exhaustive) {
                seq = vload(&p.topk.thr->seq);
                if (p.topk.ext) eseq = vload(&p.topk.ext->seq);
                read_thresholds(p.topk, s_thr);
                if (cuts) lim = cut_limit(s_thr, x, v);
            }
            s_cut[0] = lim;
            s_skip = cuts && p.lat_lb && (long long)p.lat_lb[v] >= lim;   // its landmark bound stops it
            bm[v >> 5] = 1u << (v & 31);   // the bitmap is clean: no other bit of this word is set
            sq[0] = v;
            s_qn[0] = 1; s_qn[1] = 0;
            s_ds[0] = deg; s_ds[1] = 0;
            s_lo = s_hi = v >> 5;
        }
        __syncthreads();
        u32 d = 0, nd = 1, a = 0, b = 1, c = 2;   // a, b, c: d, d+1, d+2 mod 3
        u64 f = 0;
        u32 lo = 0xffffffffu, hi = 0;             // bitmap words this thread set (global bitmap)
        int end = deg == 0 ? 1 : s_skip ? 2 : 0;   // 1 complete, 2 cut, 3 deferred
        if (ctl && deg == 0 && p.trace_lanes) lane_level(p, v, 0, 0, 1, 0);
        while (!end) {
            const u32 cnt = s_qn[a], dg = s_ds[a];
            const u32 g = dg - (d ? foot * cnt : 0u);
            if (d) {
                if (cnt == 0) { end = 1; --d; break; }
                nd += cnt;
                f += (u64)d * cnt;
            }
            // (the count itself, final since the barrier, says whether the
            // queue overflowed: every thread leaves at the same level)
            if (cnt > p.sparse_qcap) { end = 3; break; }
            if (ctl && p.trace_lanes) lane_level(p, v, d, f, nd, g);
            if ((long long)(f - g) + (long long)(d + 2) * ((long long)x - nd) >= s_cut[d & 1]) { end = 2; break; }
            u64 nseq = 0, neseq = 0;
            if (ctl) {
                s_qn[c] = 0;
                s_ds[c] = 0;
                s_st[ST_MVIS] += dg;
                s_st[ST_ENTRIES] += cnt;
                if (cuts) {
                    nseq = vload(&p.topk.thr->seq);
                    if (p.topk.ext) neseq = vload(&p.topk.ext->seq);
                }
            }
            const u32* qc = (d & 1) ? sq + kLatQueue : sq;
            u32* qn = (d & 1) ? sq : sq + kLatQueue;
            const u32* gqc = gq + (d & 1) * (size_t)gstride;
            u32* gqn = gq + ((d & 1) ^ 1) * (size_t)gstride;
            u32 dsum = 0;
            for (u32 e0 = wid * 32; e0 < cnt; e0 += THREADS) {
                const u32 e = e0 + lane;
                u32 r[RW];
#pragma unroll
                for (int j = 0; j < RW; ++j) r[j] = v;   // no entry: a visited vertex
                if (e < cnt) {
                    const u32 u = (e < kLatQueue ? qc[e] : __ldcg(&gqc[e])) & kLatIdMask;
                    load_row<RW>(rows, u, r);
                }
                u32 w[RW];
#pragma unroll
                for (int j = 0; j < RW; ++j) {
                    const u32 i = (r[j] & kLatIdMask) >> 5;
                    w[j] = SMEM ? bm[i] : __ldcg(&bm[i]);
                }
                u32 found = 0;   // how many of the row's entries this thread discovered
#pragma unroll
                for (int j = 0; j < RW; ++j) {
                    const u32 i = (r[j] & kLatIdMask) >> 5;
                    const u32 seen = __funnelshift_r(w[j], 0, r[j]) & 1u;
                    const u32 old = set_if_clear<SMEM>(&bm[i], __funnelshift_l(0, 1u, r[j]), seen);
                    w[j] = ~__funnelshift_r(old, 0, r[j]) & 1u;   // 1: discovered
                    found += w[j];
                    dsum += (r[j] >> 28) * w[j];
                    if (!SMEM && w[j]) { lo = min(lo, i); hi = max(hi, i); }
                }
                u32 off, total;
                warp_places<RW>(found, off, total);
                if (total) {
                    u32 at = 0;
                    if (lane == 0) at = atomicAdd(&s_qn[b], total);
                    at = __shfl_sync(0xffffffffu, at, 0);
                    u32 k = at + off;
                    if (at + total <= kLatQueue) {
#pragma unroll
                        for (int j = 0; j < RW; ++j) {
                            if (w[j]) qn[k] = r[j];
                            k += w[j];
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < RW; ++j) {
                            if (w[j]) {
                                if (k < kLatQueue) qn[k] = r[j];
                                else if (k < p.sparse_qcap) gqn[k] = r[j];
                            }
                            k += w[j];
                        }
                    }
                }
            }
            dsum = __reduce_add_sync(0xffffffffu, dsum);
            if (lane == 0 && dsum) atomicAdd(&s_ds[b], dsum);
            if (ctl && cuts) {
                long long lim = s_cut[d & 1];
                if (nseq != seq || neseq != eseq) {
                    seq = nseq; eseq = neseq;
                    read_thresholds(p.topk, s_thr);
                    lim = cut_limit(s_thr, x, v);
                }
                s_cut[(d & 1) ^ 1] = lim;
            } else if (ctl) {
                s_cut[(d & 1) ^ 1] = s_cut[d & 1];
            }
            __syncthreads();
            const u32 t = a; a = b; b = c; c = t;
            ++d;
        }
        // the source's footprint: the whole bitmap in shared memory (a few
        // stores per thread), the range of words it set in global memory
        if (SMEM) {
            __syncthreads();   // the last level's reads of the bitmap and the shared state
            for (u32 i = tid; i < (words + 3) / 4; i += THREADS) ((uint4*)bm)[i] = make_uint4(0, 0, 0, 0);
        } else {
            lo = __reduce_min_sync(0xffffffffu, lo);
            hi = __reduce_max_sync(0xffffffffu, hi);
            if (lane == 0 && lo <= hi) { atomicMin(&s_lo, lo); atomicMax(&s_hi, hi); }
            __syncthreads();
            const u32 wl = s_lo, wh = s_hi;
            for (u32 i = wl + tid; i <= wh; i += THREADS) bm[i] = 0;
            if (ctl) s_st[ST_CLEARED] += wh - wl + 1;
        }
        if (ctl) {
            if (SMEM) s_st[ST_CLEARED] += words;
            s_st[ST_DISC] += nd - 1;
            const u32 levels = end == 1 && deg ? d + 1 : d;   // levels expanded
            s_st[ST_LEVELS] += levels;
            if (levels > s_st[ST_MAXLEVEL]) s_st[ST_MAXLEVEL] = levels;
            if (end == 1) {
                s_st[ST_COMPLETED]++;
                if (p.trace_lanes) lane_end(p, v, d, f, nd, false);
                if (p.exhaustive) {
                    p.out_far[v] = f;
                    p.out_reach[v] = nd;
                } else {
                    lattice_complete(p, s_thr, v, f, nd);
                }
            } else if (end == 2) {
                s_st[ST_CUT]++;
                if (p.trace_lanes) lane_end(p, v, d, f, nd, true);
            } else {
                // the frontier outgrew its queue: the source goes to the
                // grid-wide pass (where none follows, the run fails)
                if (p.defer_src) {
                    p.defer_src[atomicAdd(p.defer_n, 1u)] = v;
                    s_st[ST_DEFERRED]++;
                } else {
                    atomicOr(p.err, DEV_ERR_TABLE_FULL);
                }
            }
        }
    }
    if (ctl) {
        s_st[ST_ARCWORDS] = s_st[ST_MVIS];
        s_st[ST_DISCWORDS] = s_st[ST_DISC];
        for (int i = 0; i < ST_COUNT; ++i) {
            if (i == ST_MAXLEVEL) atomicMax(&p.stats[i], s_st[i]);
            else if (s_st[i]) atomicAdd(&p.stats[i], s_st[i]);
        }
    }
}

// ------------------------------------------------------------- launchers
// Threads per CTA by default: about one per vertex of an average frontier,
// which on a lattice is somewhat below sqrt(n) (128^2 at 64 / 256 threads: 2.7
// / 3.3 ms; 512^2 at 128 / 256: 417 / 389).  From 2^19 vertices the bitmap
// leaves room for one or two CTAs per SM, and 1024 threads are best (1/16 of
// 1024^2: 256 threads 1,007 ms, 1024 731); with the bitmap in global memory
// 256 again (1,087 ms against 1,239 at 512).
int lattice_threads(uint32_t n) {
    return n <= (1u << 15) ? 64 : n <= (1u << 17) ? 128 : n <= (1u << 19) || !lattice_smem(n) ? 256 : 1024;
}

typedef void (*LatKernel)(WaveParams);

template <int T>
static LatKernel lat_pick(int rw, bool smem) {
    if (rw == 4) return smem ? k_lattice<T, 4, true> : k_lattice<T, 4, false>;
    return smem ? k_lattice<T, 8, true> : k_lattice<T, 8, false>;
}

static LatKernel lat_kernel(int threads, int rw, bool smem) {
    switch (threads) {
        case 64: return lat_pick<64>(rw, smem);
        case 128: return lat_pick<128>(rw, smem);
        case 256: return lat_pick<256>(rw, smem);
        case 512: return lat_pick<512>(rw, smem);
        case 1024: return lat_pick<1024>(rw, smem);
        default: return nullptr;
    }
}

int lattice_blocks_per_sm(uint32_t n, int threads, int rw) {
    LatKernel k = lat_kernel(threads, rw, lattice_smem(n));
    if (!k) return 0;
    const size_t dyn = lattice_dyn_smem(n);
    if (cudaFuncSetAttribute((const void*)k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)lattice_dyn_smem(kLatSmemMaxN)) != cudaSuccess)
        return 0;
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, (const void*)k, threads, dyn) != cudaSuccess) return 0;
    return per;
}

int launch_lattice(const WaveParams& p, int rw, int blocks, int threads, cudaStream_t s) {
    LatKernel k = lat_kernel(threads, rw, lattice_smem(p.g.n));
    if (!k) return -2;
    k<<<blocks, threads, lattice_dyn_smem(p.g.n), s>>>(p);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace bcm
