// Farness and reach of every vertex by complete BFS, for graphs whose bit
// planes stay in L2 (bcm_farness_all, bcm_farness_all_noalloc), and the top-k
// of small graphs from them.
//
// The lanes of a wave are targets, not sources: bit j of vis[x] says that x
// reaches target t_j.  A level then is a pull over out-arcs,
//     new(x) = alive & ~vis(x) & (OR over arcs x -> u of F(u)),
// F(u) the lanes that u gained at the level before, and x's own thread adds
// d popc(new) to f(x) and popc(new) to r(x).  So nothing is counted per lane
// (the grid-wide kernel transposes 32 x 32 bit blocks for that), no in-arc
// CSR is needed on digraphs, there are no frontier lists, and no atomics
// inside a level.  A lane that gained nothing in a level is dead.
//
// A wave of 64 W targets belongs to a cluster of C CTAs (a hardware cluster
// barrier per level); the clusters take waves from a counter.  Planes of 24 n W
// bytes per cluster: C is chosen so that those of all clusters fit in L2
// together and no SM is idle.
//
// What bounds it: the latency of the gathers of F (one L2 sector per arc and
// level until x has all lanes; Chung-Lu 2^14: long-scoreboard stalls 16 of 28
// cycles per issue, L1 60% busy, issue 24%): farness of every vertex, grid-wide
// kernel -> here: Chung-Lu 2^14 36.6 -> 0.74 ms, R-MAT 2^16 103 -> 12.5; without
// allocation (in-arcs unknown, level 1 pulled) Chung-Lu 10,007 5.3 -> 0.6 ms.
#include <cuda_runtime.h>

#include "internal.h"

namespace bcm {

constexpr int kApThreads = 1024;
constexpr u32 kApRow = 32;       // longer rows are scanned by a warp
constexpr u32 kApBig = 4096;     // ... by a CTA

__device__ __forceinline__ void ap_barrier(int C) {
    if (C == 1) __syncthreads();
    else asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Loads of the planes: through L2 where another CTA of the cluster may have
// written them.
template <int W, int C>
__device__ __forceinline__ void ap_load(const u64* p, u64 (&w)[W]) {
    if (W == 1) {
        w[0] = C == 1 ? *p : __ldcg(p);
    } else {
#pragma unroll
        for (int i = 0; i < W; i += 2) {
            const ulonglong2 t = C == 1 ? *(const ulonglong2*)(p + i) : __ldcg((const ulonglong2*)(p + i));
            w[i] = t.x;
            w[i + 1] = t.y;
        }
    }
}
template <int W>
__device__ __forceinline__ void ap_store(u64* p, const u64 (&w)[W]) {
    if (W == 1) {
        p[0] = w[0];
    } else {
#pragma unroll
        for (int i = 0; i < W; i += 2) *(ulonglong2*)(p + i) = make_ulonglong2(w[i], w[i + 1]);
    }
}

// Rows with more than `deg` arcs: the first ones (rows by degree descending).
__device__ __forceinline__ u32 rows_over(const u32* rp, u32 n, u32 deg) {
    u32 lo = 0, hi = n;
    while (lo < hi) {
        const u32 mid = (lo + hi) >> 1;
        if (__ldg(&rp[mid + 1]) - __ldg(&rp[mid]) > deg) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// What row x gained at level d: its words, its sums, and the lanes it gained.
template <int W>
__device__ __forceinline__ void ap_finish(u64* vis, u64* Fn, u64* acc, u32 x, u32 d, u64 accx, u64 (&v)[W],
                                          const u64 (&pend)[W], u64 (&got)[W], u64 (&gain)[W]) {
    u32 c = 0;
#pragma unroll
    for (int g = 0; g < W; ++g) {
        got[g] &= pend[g];
        gain[g] |= got[g];
        v[g] |= got[g];
        c += __popcll(got[g]);
    }
    ap_store<W>(&Fn[(size_t)x * W], got);
    if (c) {
        ap_store<W>(&vis[(size_t)x * W], v);
        acc[x] = accx + ((u64)c << 32) + (u64)d * c;
    }
}

// A level sweeps every row, whatever it gains, so on graphs whose searches are
// thin (long chains, rings, many small parts) k_wave_cta is faster, which scans
// frontiers only: without allocation, 65,536 vertices in paths of ten took 11.6
// ms against its 2.9, a ring of 60,000 and 40 arcs each 20.9 s against 4.5.  No
// count that is known beforehand tells such graphs apart, so there (kApPaced) the
// first waves compare their pace with what that kernel takes for a level,
// kRivalLevelNs and kRivalFoundNs for each (vertex, lane) pair that it reaches
// (within a third of what it took on paths, cycles, rings and chains of 8,000 to
// 130,000 vertices; on power-law graphs, where all pairs is 10 to 30 times
// faster, it takes a tenth of that).  They look at levels 32, 64, 128, ... and at
// their ends, and give up once half of the clusters have looked and the pace is
// worse by a tenth -- by two before level 256, since frontiers that widen have
// little at first (directed grids of 128^2 and 300^2: all pairs 5.7 and 725 ms,
// k_wave_cta 45 and 3,140).  Where both take about the same the choice can be
// wrong by a quarter.
constexpr u64 kRivalLevelNs = 4000, kRivalFoundNs = 30;
constexpr u32 kApQuit = 24;      // lanes: past [3][2W], three rotating copies of Pace::quit

// kApSorted: p.vertex.  kApGiven: rows in any order.  kApPaced: either, p.pace.
enum ApKind { kApSorted, kApGiven, kApPaced };

// Rows are numbered by degree descending where the caller laid them out so
// (p.vertex: the vertex of each row): a warp's 32 rows then have about the
// same length, and the few long ones come first.
template <int W, int C, ApKind KIND>
__global__ void __launch_bounds__(kApThreads) k_allpairs(AllPairs p) {
    constexpr bool PACED = KIND == kApPaced;
    __shared__ u32 s_or[2 * W];          // lanes that gained a row, this CTA's part
    __shared__ unsigned long long s_acc[W];
    __shared__ unsigned long long s_st, s_found;
    // (PACED; thread 0's: when and where this wave was looked at last, what its CTA's rows had then)
    __shared__ u64 s_look_ns, s_look_found;
    __shared__ u32 s_look_d;
    const u32 tid = threadIdx.x, lane = tid & 31;
    const u32 rank = blockIdx.x % C, cl = blockIdx.x / C, ncl = gridDim.x / C;
    const u32 n = p.n;
    constexpr u32 NW = kApThreads / 32 * C;                 // warps of the cluster
    constexpr int U = W == 4 ? 2 : 4;                       // arcs in flight per thread (registers)
    const u32 gw = (tid >> 5) * C + rank;                   // numbered across its CTAs first
    char* slot = p.slots + (size_t)cl * p.slot_stride;
    u64* const vis = (u64*)slot;
    u64* const F0 = vis + (size_t)n * W;
    u64* const F1 = F0 + (size_t)n * W;
    u64* const acc = F1 + (size_t)n * W;                    // per row: count << 32 | distance sum
    u32* const gor = p.lanes + (size_t)cl * (3 * 2 * 8);    // [3][2W] the cluster's lanes that gained a row
    const u32 waves = (n + 64 * W - 1) / (64 * W);
    // (unsorted rows: every row is scanned by a thread or, past kApRow, a warp)
    const u32 nbig = p.vertex ? rows_over(p.rp, n, kApBig) : 0;
    const u32 nwide = p.vertex ? rows_over(p.rp, n, kApRow) : n;
    if (tid == 0) { s_st = 0; s_found = 0; }
    u64 mvis = 0;
    u32 levels = 0, maxlev = 0;
    bool quit = false;
    // level d of a wave has ended; `found`: the pairs this thread's rows have
    auto look = [&](u32 d, u64 found) {
        for (int o = 16; o; o >>= 1) found += __shfl_xor_sync(0xffffffffu, found, o);
        if (lane == 0 && found) atomicAdd(&s_found, (unsigned long long)found);
        __syncthreads();
        if (tid == 0) {
            atomicAdd(&p.pace->found, (unsigned long long)(s_found - s_look_found));
            s_look_found = s_found;
            s_found = 0;
            if (rank == 0) {
                const u64 now = global_ns(), dt = now - s_look_ns, dl = d - s_look_d;
                s_look_ns = now;
                s_look_d = d;
                const u64 ns = atomicAdd(&p.pace->ns, (unsigned long long)dt) + dt;
                const u64 lv = atomicAdd(&p.pace->levels, (unsigned long long)dl) + dl;
                const u32 looks = atomicAdd(&p.pace->looks, 1u) + 1;
                // time left in rounds of waves, this kernel's and the other's
                const u64 mine = ns * ((waves + ncl - 1) / ncl);
                const u64 other = (kRivalLevelNs * lv + kRivalFoundNs * vload(&p.pace->found) / W) * p.rival_rounds;
                if (looks * 2 >= ncl && mine * 10 > other * (d < 256 ? 20 : 11)) vstore(&p.pace->quit, 1u);
            }
        }
    };
    for (u32 wave = cl; wave < waves; wave += ncl) {
        // (looked at, the first waves have to speak for all: where there are many, they are spread over the targets)
        const u32 t0 = (PACED ? (u32)((u64)wave * p.wave_step % waves) : wave) * 64 * W;
        const u32 nt = n - t0 < 64u * W ? n - t0 : 64u * W;
        u64 alive[W];
#pragma unroll
        for (int g = 0; g < W; ++g) {
            const u32 left = nt > 64u * g ? nt - 64u * g : 0u;
            alive[g] = left >= 64 ? ~0ull : ((1ull << left) - 1);
        }
        for (u32 x = gw * 32 + lane; x < n; x += NW * 32) {
            const bool own = x >= t0 && x - t0 < nt;
            u64 w[W];
#pragma unroll
            for (int g = 0; g < W; ++g) w[g] = own && (x - t0) / 64 == (u32)g ? 1ull << ((x - t0) & 63) : 0;
            ap_store<W>(&vis[(size_t)x * W], w);
            ap_store<W>(&F0[(size_t)x * W], w);
            acc[x] = own ? 1ull << 32 : 0;
            if (p.rrp) {
#pragma unroll
                for (int g = 0; g < W; ++g) w[g] = 0;
                ap_store<W>(&F1[(size_t)x * W], w);
            }
        }
        if (rank == 0 && tid < 3 * 2 * W) gor[tid] = 0;
        if (tid < 2 * W) s_or[tid] = 0;
        ap_barrier(C);
        if (PACED && tid == 0) {
            s_look_ns = global_ns();
            s_look_found = 0;
            s_look_d = 0;
        }
        // level 1 by push where the in-arcs are there: the targets' few rows
            // instead of every arc of the graph (half to four fifths of all
            // the arcs a wave's pulls would scan)
        if (p.rrp) {
            for (u32 j = rank; j < nt; j += C) {            // long rows: the CTA
                const u32 v = p.vertex[t0 + j], b = __ldg(&p.rrp[v]), e = __ldg(&p.rrp[v + 1]);
                if (e - b <= 512) break;                    // (by degree: no longer one follows, but see below)
                for (u32 i = b + tid; i < e; i += kApThreads)
                    atomicOr(&F1[(size_t)__ldg(&p.pos[__ldg(&p.rcol[i])]) * W + (j >> 6)], 1ull << (j & 63));
            }
            // the CTA stopped at its first short row; in-degrees need not
            // follow the rows' order, so a warp takes every row from there on
            u32 first = rank;
            while (first < nt) {
                const u32 v = p.vertex[t0 + first];
                if (__ldg(&p.rrp[v + 1]) - __ldg(&p.rrp[v]) <= 512) break;
                first += C;
            }
            for (u32 j = first + (tid >> 5) * C; j < nt; j += NW) {
                const u32 v = p.vertex[t0 + j], b = __ldg(&p.rrp[v]), e = __ldg(&p.rrp[v + 1]);
                for (u32 i = b + lane; i < e; i += 32)
                    atomicOr(&F1[(size_t)__ldg(&p.pos[__ldg(&p.rcol[i])]) * W + (j >> 6)], 1ull << (j & 63));
            }
            ap_barrier(C);
        }
        u32 par = 0, d = 1;
        for (;; ++d) {
            const bool pushed = d == 1 && p.rrp;   // F1 already holds every row's gathered word
            const u64* Fc = (d & 1) ? F0 : F1;
            u64* Fn = (d & 1) ? F1 : F0;
            u64 gain[W];
#pragma unroll
            for (int g = 0; g < W; ++g) gain[g] = 0;
            // the longest rows, one CTA each
            for (u32 x = rank; x < (pushed ? 0u : nbig); x += C) {
                if (tid < W) s_acc[tid] = 0;
                __syncthreads();
                const u32 b = __ldg(&p.rp[x]), e = __ldg(&p.rp[x + 1]);
                u64 f[W];
#pragma unroll
                for (int g = 0; g < W; ++g) f[g] = 0;
                for (u32 i = b + tid; i < e; i += kApThreads) {
                    u64 w[W];
                    ap_load<W, C>(&Fc[(size_t)__ldg(&p.col[i]) * W], w);
#pragma unroll
                    for (int g = 0; g < W; ++g) f[g] |= w[g];
                }
#pragma unroll
                for (int g = 0; g < W; ++g) {
                    const u32 l = __reduce_or_sync(0xffffffffu, (u32)f[g]);
                    const u32 h = __reduce_or_sync(0xffffffffu, (u32)(f[g] >> 32));
                    if (lane == 0 && (l | h)) atomicOr(&s_acc[g], ((u64)h << 32) | l);
                }
                __syncthreads();
                if (tid == 0) {
                    u64 v[W], pend[W], got[W];
                    ap_load<W, C>(&vis[(size_t)x * W], v);
#pragma unroll
                    for (int g = 0; g < W; ++g) {
                        pend[g] = alive[g] & ~v[g];
                        got[g] = s_acc[g];
                    }
                    ap_finish<W>(vis, Fn, acc, x, d, C == 1 ? acc[x] : __ldcg(&acc[x]), v, pend, got, gain);
                }
                __syncthreads();
            }
            // long rows, one warp each
            auto wide_row = [&](u32 x) {
                u64 v[W], pend[W], got[W];
                ap_load<W, C>(&vis[(size_t)x * W], v);
                const u32 b = __ldg(&p.rp[x]), e = __ldg(&p.rp[x + 1]);
                bool any = false;
#pragma unroll
                for (int g = 0; g < W; ++g) {
                    pend[g] = alive[g] & ~v[g];
                    got[g] = 0;
                    any = any || pend[g] != 0;
                }
                for (u32 i = b; any && i < e; i += 32 * U) {
                    u64 f[W];
#pragma unroll
                    for (int g = 0; g < W; ++g) f[g] = 0;
                    u32 u[U];
#pragma unroll
                    for (int j = 0; j < U; ++j) {
                        const u32 a = i + 32 * j + lane;
                        u[j] = __ldg(&p.col[a < e ? a : e - 1]);
                    }
#pragma unroll
                    for (int j = 0; j < U; ++j) {
                        u64 w[W];
                        ap_load<W, C>(&Fc[(size_t)u[j] * W], w);
#pragma unroll
                        for (int g = 0; g < W; ++g) f[g] |= w[g];
                    }
                    any = false;
#pragma unroll
                    for (int g = 0; g < W; ++g) {
                        const u64 m = f[g] & pend[g];
                        const u32 l = __reduce_or_sync(0xffffffffu, (u32)m);
                        const u32 h = __reduce_or_sync(0xffffffffu, (u32)(m >> 32));
                        got[g] |= ((u64)h << 32) | l;
                        any = any || (pend[g] & ~got[g]) != 0;
                    }
                }
                if (lane == 0) {
                    ap_finish<W>(vis, Fn, acc, x, d, C == 1 ? acc[x] : __ldcg(&acc[x]), v, pend, got, gain);
                }
                __syncwarp();
            };
            if (KIND != kApSorted && !p.vertex) {
                // unsorted rows: a warp looks over 32 at a time (one at a time
                // the lengths alone took 28 us a level at n = 8,000)
                for (u32 x0 = gw * 32; x0 < (pushed ? 0u : n); x0 += NW * 32) {
                    const u32 y = x0 + lane;
                    u32 todo = __ballot_sync(0xffffffffu, y < n && __ldg(&p.rp[y + 1]) - __ldg(&p.rp[y]) > kApRow);
                    for (; todo; todo &= todo - 1) wide_row(x0 + __ffs(todo) - 1);
                }
            } else {
                for (u32 x = nbig + gw; x < (pushed ? 0u : nwide); x += NW) wide_row(x);
            }
            // the others, one thread each; where the rows are sorted, a warp's 32
            // rows lie interleaved (entry j of lane l at 32 j + l, padded to the
            // first one's length with the row itself, which adds nothing): one
            // line per load instead of 32, and the loads of row entries are half
            // of all the loads
            for (u32 x0 = (p.vertex && !pushed ? nwide : 0) + gw * 32; x0 < n; x0 += NW * 32) {
                const u32 x = x0 + lane;
                if (x >= n) continue;
                u64 v[W], pend[W], got[W];
                ap_load<W, C>(&vis[(size_t)x * W], v);
                const u64 accx = C == 1 ? acc[x] : __ldcg(&acc[x]);
                bool any = false;
#pragma unroll
                for (int g = 0; g < W; ++g) {
                    pend[g] = alive[g] & ~v[g];
                    got[g] = 0;
                    any = any || pend[g] != 0;
                }
                if (pushed) {
                    ap_load<W, 8>(&Fn[(size_t)x * W], got);   // (atomics wrote them: through L2)
                } else if (p.vertex) {
                    const u32 b = __ldg(&p.rp[x0]), len = __ldg(&p.rp[x0 + 1]) - b;
                    const u32* at = p.col + b + lane;
                    for (u32 i = 0; any && i < len; i += U) {
                        u32 u[U];
#pragma unroll
                        for (int j = 0; j < U; ++j) u[j] = __ldg(&at[32 * (i + j < len ? i + j : len - 1)]);
#pragma unroll
                        for (int j = 0; j < U; ++j) {
                            u64 w[W];
                            ap_load<W, C>(&Fc[(size_t)u[j] * W], w);
#pragma unroll
                            for (int g = 0; g < W; ++g) got[g] |= w[g];
                        }
                        any = false;
#pragma unroll
                        for (int g = 0; g < W; ++g) any = any || (pend[g] & ~got[g]) != 0;
                    }
                } else {
                    const u32 b = __ldg(&p.rp[x]), e = __ldg(&p.rp[x + 1]);
                    if (e - b > kApRow) continue;   // a warp had it
                    for (u32 i = b; any && i < e; ++i) {
                        u64 w[W];
                        ap_load<W, C>(&Fc[(size_t)__ldg(&p.col[i]) * W], w);
                        any = false;
#pragma unroll
                        for (int g = 0; g < W; ++g) {
                            got[g] |= w[g];
                            any = any || (pend[g] & ~got[g]) != 0;
                        }
                    }
                }
                ap_finish<W>(vis, Fn, acc, x, d, accx, v, pend, got, gain);
            }
            // lanes that gained a row live on
            __syncwarp();
#pragma unroll
            for (int g = 0; g < W; ++g) {
                const u32 l = __reduce_or_sync(0xffffffffu, (u32)gain[g]);
                const u32 h = __reduce_or_sync(0xffffffffu, (u32)(gain[g] >> 32));
                if (lane == 0 && l) atomicOr(&s_or[2 * g], l);
                if (lane == 0 && h) atomicOr(&s_or[2 * g + 1], h);
            }
            __syncthreads();
            u32* const go = gor + par * 2 * W;
            if (tid < 2 * W) {
                if (s_or[tid]) atomicOr(&go[tid], s_or[tid]);
                s_or[tid] = 0;
                // the next level's copy: last read two levels ago
                if (rank == 0) gor[((par + 1) % 3) * 2 * W + tid] = 0;
            }
            if (PACED && rank == 0 && tid == 0) gor[kApQuit + par] = vload(&p.pace->quit);
            ap_barrier(C);
            u64 live = 0;
#pragma unroll
            for (int g = 0; g < W; ++g) {
                alive[g] &= ((u64)__ldcg(&go[2 * g + 1]) << 32) | __ldcg(&go[2 * g]);
                live |= alive[g];
            }
            if (PACED) quit = __ldcg(&gor[kApQuit + par]) != 0;   // (the same for the whole cluster)
            par = (par + 1) % 3;
            if (!live || quit) break;
            if (PACED && wave < ncl && d >= 32 && !(d & (d - 1))) {
                u64 found = 0;
                for (u32 x = gw * 32 + lane; x < n; x += NW * 32) found += __ldcg(&acc[x]) >> 32;
                look(d, found);
            }
        }
        if (quit) break;
        if (rank == 0 && tid == 0) { levels += d; maxlev = d > maxlev ? d : maxlev; }
        // this wave's share of every vertex's farness and reach, and of the
        // arcs a search per source would scan (deg(t) for each x that reaches
        // t): counts of the columns, most of which are full or empty
        u64 found = 0;
        for (u32 x0 = gw * 32; x0 < n; x0 += NW * 32) {
            const u32 x = x0 + lane;
            u64 v[W];
#pragma unroll
            for (int g = 0; g < W; ++g) v[g] = 0;
            if (x < n) {
                ap_load<W, C>(&vis[(size_t)x * W], v);
                const u64 a = C == 1 ? acc[x] : __ldcg(&acc[x]);
                if (PACED) found += a >> 32;
                if (a) {
                    const u32 y = p.vertex ? __ldg(&p.vertex[x]) : x;
                    atomicAdd(&p.far[y], (unsigned long long)(a & 0xffffffffull));
                    atomicAdd(&p.reach[y], (u32)(a >> 32));
                }
            }
#pragma unroll
            for (int h = 0; h < 2 * W; ++h) {
                const u32 m = (u32)(v[h / 2] >> (32 * (h & 1)));
                const u32 full = __reduce_and_sync(0xffffffffu, m);
                u32 mix = __reduce_or_sync(0xffffffffu, m) & ~full;
                u32 c = (full >> lane) & 1u ? 32u : 0u;   // lane j: target t0 + 32 h + j
                while (mix) {
                    const int j = __ffs(mix) - 1;
                    mix &= mix - 1;
                    const u32 k = __popc(__ballot_sync(0xffffffffu, (m >> j) & 1u));
                    if (lane == (u32)j) c = k;
                }
                const u32 t = t0 + 32 * h + lane;
                if (c) {
                    const u32 y = p.vertex ? __ldg(&p.vertex[t]) : t;
                    mvis += (u64)c * (__ldg(&p.grp[y + 1]) - __ldg(&p.grp[y]));
                }
            }
        }
        // (a wave to come, and most of them: else it is too late to give up)
        if (PACED && wave + ncl < waves && (wave < ncl || wave * 4 < waves)) look(d, found);
        ap_barrier(C);
    }
    for (int o = 16; o; o >>= 1) mvis += __shfl_xor_sync(0xffffffffu, mvis, o);
    if (lane == 0 && mvis) atomicAdd(&s_st, (unsigned long long)mvis);
    __syncthreads();
    if (tid == 0) {
        if (s_st) {
            atomicAdd(&p.stats[ST_MVIS], s_st);
            atomicAdd(&p.stats[ST_ARCWORDS], s_st / (64 * W));
        }
        if (rank == 0 && levels) {
            atomicAdd(&p.stats[ST_LEVELS], (unsigned long long)levels);
            atomicMax(&p.stats[ST_MAXLEVEL], (unsigned long long)maxlev);
        }
        if (blockIdx.x == 0) {
            atomicAdd(&p.stats[ST_COMPLETED], (unsigned long long)n);
            atomicAdd(&p.stats[ST_WAVES], (unsigned long long)waves);
        }
    }
}

// ------------------------------------------------ rows by degree descending
// Row i is that of vertex order[i], neighbours are row numbers (pos: the row
// of each vertex).  Rows over kApRow are plain; from the first shorter one on,
// groups of 32 rows are interleaved and padded to their first row's length
// (at most 32 * 32 entries more in all, the lengths descending).
__device__ __forceinline__ u32 degree_of(const u32* grp, const u32* order, u32 i) {
    const u32 v = __ldg(&order[i]);
    return __ldg(&grp[v + 1]) - __ldg(&grp[v]);
}

__device__ __forceinline__ u32 first_narrow(const u32* grp, const u32* order, u32 n) {
    u32 lo = 0, hi = n;
    while (lo < hi) {
        const u32 mid = (lo + hi) >> 1;
        if (degree_of(grp, order, mid) > kApRow) lo = mid + 1; else hi = mid;
    }
    return lo;
}

__global__ void k_rows_degree(const u32* grp, const u32* order, u32 n, u32* len, u32* pos) {
    const u32 stride = gridDim.x * blockDim.x, nw = first_narrow(grp, order, n);
    for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += stride) {
        if (i == n) { len[n] = 0; break; }
        len[i] = degree_of(grp, order, i < nw ? i : nw + ((i - nw) & ~31u));
        pos[__ldg(&order[i])] = i;
    }
}

__global__ void k_rows_copy(const u32* grp, const u32* gcol, const u32* order, const u32* pos, u32 n, const u32* rp,
                            u32* col) {
    const u32 lane = threadIdx.x & 31, nwarps = gridDim.x * blockDim.x / 32, nw = first_narrow(grp, order, n);
    for (u32 i = (blockIdx.x * blockDim.x + threadIdx.x) / 32; i < n; i += nwarps) {
        const u32 v = __ldg(&order[i]), g = __ldg(&grp[v]), deg = __ldg(&grp[v + 1]) - g, len = rp[i + 1] - rp[i];
        const u32 f = i < nw ? i : nw + ((i - nw) & ~31u);   // the group's first row
        const u32 b = rp[f] + (i - f), step = i < nw ? 1 : 32;
        for (u32 j = lane; j < len; j += 32) col[b + j * step] = j < deg ? pos[gcol[g + j]] : i;
    }
}

static size_t sorted_col_offset(uint32_t n) { return al256(((size_t)n + 1) * 4); }
static size_t sorted_pos_offset(uint32_t n, uint64_t m) { return sorted_col_offset(n) + al256((size_t)m * 4 + 2048 * 4); }
size_t sorted_rows_bytes(uint32_t n, uint64_t m) { return sorted_pos_offset(n, m) + al256((size_t)n * 4); }
size_t sorted_rows_scratch_bytes(uint32_t n) { return scan_scratch_bytes((size_t)n + 1); }

void sorted_rows_use(AllPairs* a, const void* rows, uint64_t m, const uint32_t* order) {
    a->rp = (const uint32_t*)rows;
    a->col = (const uint32_t*)((const char*)rows + sorted_col_offset(a->n));
    a->pos = (const uint32_t*)((const char*)rows + sorted_pos_offset(a->n, m));
    a->vertex = order;
}

int launch_sorted_rows(const uint32_t* grp, const uint32_t* gcol, const uint32_t* order, uint32_t n, uint64_t m,
                       void* rows, void* scratch, cudaStream_t s) {
    uint32_t* rp = (uint32_t*)rows;
    uint32_t* col = (uint32_t*)((char*)rows + sorted_col_offset(n));
    uint32_t* pos = (uint32_t*)((char*)rows + sorted_pos_offset(n, m));
    const unsigned b = (n + 256) / 256 < 1216 ? (n + 256) / 256 : 1216;
    k_rows_degree<<<b, 256, 0, s>>>(grp, order, n, rp, pos);
    if (exclusive_scan_u32(rp, rp, (size_t)n + 1, nullptr, scratch, s)) return -1;
    k_rows_copy<<<(n + 7) / 8 < 2432 ? (n + 7) / 8 : 2432, 256, 0, s>>>(grp, gcol, order, pos, n, rp, col);
    note_launch(2);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// ----------------------------------------------- top-k of every vertex's key
// rank(v) = the vertices that rank before v: every pair is compared, first as
// floats (both keys N / F rounded: a difference above 8 units in the last
// place decides), else exactly.  n <= kAllPairsTopkN, so 2.7 10^8 pairs at
// most; on 152 SMs that beats a sort's passes.
__global__ void __launch_bounds__(128) k_rank(const unsigned long long* far, const u32* reach, u32 n, u32* rank) {
    __shared__ u64 s_N[128], s_F[128];
    __shared__ float s_q[128];
    const u32 v = blockIdx.x * 128 + threadIdx.x;
    u64 N = 0, F = 1;
    float q = 0;
    if (v < n) {
        score_key(far[v], reach[v], N, F);
        q = __ull2float_rn(N) / __ull2float_rn(F);
    }
    u32 r = 0;
    for (u32 b = blockIdx.y * 128; b < n; b += gridDim.y * 128) {
        const u32 u = b + threadIdx.x;
        __syncthreads();
        if (u < n) {
            u64 a, c;
            score_key(far[u], reach[u], a, c);
            s_N[threadIdx.x] = a;
            s_F[threadIdx.x] = c;
            s_q[threadIdx.x] = __ull2float_rn(a) / __ull2float_rn(c);
        }
        __syncthreads();
        const u32 cnt = n - b < 128 ? n - b : 128;
        const float hi = q * (1 + 1e-6f), lo = q * (1 - 1e-6f);
        for (u32 i = 0; i < cnt; ++i) {
            const float t = s_q[i];
            if (t > hi) ++r;
            else if (t >= lo && b + i != v) r += ranks_before(s_N[i], s_F[i], b + i, N, F, v);
        }
    }
    if (v < n && r) atomicAdd(&rank[v], r);
}

__global__ void k_emit(const unsigned long long* far, const u32* reach, const u32* rank, u32 n, TopK T) {
    const u32 v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n) return;
    const u32 r = rank[v];
    if (r < T.k) {
        T.id[r] = v;
        T.f[r] = far[v];
        T.r[r] = reach[v];
    }
    if (r + 1 == (T.k < n ? T.k : n)) {
        *T.count = r + 1;
        if (r + 1 == T.k) {   // the k-th key: bcm_topk_threshold may read it meanwhile
            u64 N, F;
            score_key(far[v], reach[v], N, F);
            threshold_publish(T.thr, N, F, v);
        }
    }
}

// ------------------------------------------------------------- launchers
template <int W, ApKind KIND>
static const void* ap_kernel(int C) {
    return C == 1 ? (const void*)k_allpairs<W, 1, KIND> : C == 2 ? (const void*)k_allpairs<W, 2, KIND>
         : C == 4 ? (const void*)k_allpairs<W, 4, KIND> : (const void*)k_allpairs<W, 8, KIND>;
}

template <ApKind KIND>
static const void* ap_kernel(int W, int C) {
    return W == 1 ? ap_kernel<1, KIND>(C) : W == 2 ? ap_kernel<2, KIND>(C) : ap_kernel<4, KIND>(C);
}

int launch_allpairs(const AllPairs& p, int W, int C, int clusters, cudaStream_t s) {
    const void* k = p.pace ? ap_kernel<kApPaced>(W, C) : p.vertex ? ap_kernel<kApSorted>(W, C) : ap_kernel<kApGiven>(W, C);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(clusters * C);
    cfg.blockDim = dim3(kApThreads);
    cfg.stream = s;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = C;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    AllPairs q = p;
    void* args[] = {(void*)&q};
    const cudaError_t e = cudaLaunchKernelExC(&cfg, k, args);
    note_launch();
    return e == cudaSuccess ? 0 : -1;
}

int launch_rank_topk(const unsigned long long* far, const uint32_t* reach, uint32_t n, uint32_t* rank, const TopK& T,
                     cudaStream_t s) {
    const unsigned bx = (n + 127) / 128, by = bx >= 608 ? 1 : 608 / bx < bx ? 608 / bx : bx;
    k_rank<<<dim3(bx, by), 128, 0, s>>>(far, reach, n, rank);
    k_emit<<<(n + 255) / 256, 256, 0, s>>>(far, reach, rank, n, T);
    note_launch(2);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace bcm
