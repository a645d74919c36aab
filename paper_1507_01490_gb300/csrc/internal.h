// Internal interfaces between the library's translation units (not part of
// the C-ABI).  Kernels are launched only through the functions declared here.
#pragma once
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "common.cuh"
#include "shape.h"

namespace bcm {

// Counters accumulated by the wave kernels, in this order.
enum Stat {
    ST_MVIS = 0,        // arcs scanned, counted per source (Section 3.1's m_vis)
    ST_DISC,            // (source, vertex) discoveries
    ST_COMPLETED,       // sources whose BFS ran to the end
    ST_CUT,             // sources stopped by the bound
    ST_WAVES,           // waves run
    ST_LEVELS,          // levels expanded, summed over waves
    ST_MAXLEVEL,        // deepest level reached
    ST_ENTRIES,         // frontier words expanded (level >= 1)
    ST_ARCWORDS,        // (arc, frontier word) pairs scanned
    ST_DISCWORDS,       // frontier words created (first discovery in a level)
    ST_CLEARED,         // vertex words cleared at wave ends
    ST_DEFERRED,        // sources a per-CTA wave handed to the grid-wide pass
    ST_PULLENTRIES,     // frontier words of pulled levels (also in ST_ENTRIES)
    ST_COUNT
};

// The graph as the kernels see it.  Offsets are narrowed to 32 bits (m < 2^32).
struct GraphDev {
    uint32_t n;
    uint64_t m;
    const uint32_t* rp;      // [n+1]
    const uint32_t* col;     // [m]
    const uint32_t* order;   // [n] vertices by (degree desc, id asc)
    const uint32_t* xlo;     // [n] r(v) (undirected) or alpha(v)
    const uint32_t* xhi;     // [n] r(v) (undirected) or omega(v)
    const uint32_t* rrp;     // in-arcs CSR (the graph itself when undirected)
    const uint32_t* rcol;
};

// Per-slot working memory of one MS-BFS wave with W words (64W sources) per
// vertex, for n vertices (or table entries).  Word index of (entry v, word g)
// is v*W + g; each word has a 32-byte record (vis, key, F[0], F[1]), then two
// frontier lists and a clear log of 4-byte word indices.
constexpr size_t slot_bytes(uint32_t n, int W) {
    size_t nw = (size_t)n * W;
    size_t b = nw * (4 * sizeof(uint64_t) + 3 * sizeof(uint32_t));
    return (b + 255) & ~(size_t)255;
}

// One-source-per-CTA slot (k_sparse): a visited bitmap of one bit per vertex,
// the log of its words that became non-zero, then two queues of qcap
// entries each (a frontier vertex's first arc and degree, 8 bytes).
__host__ __device__ constexpr size_t sparse_bitmap_bytes(uint32_t n) { return al256(((size_t)n + 31) / 32 * sizeof(uint32_t)); }
__host__ __device__ constexpr size_t sparse_slot_bytes(uint32_t n, uint32_t qcap) {
    return 2 * sparse_bitmap_bytes(n) + 2 * al256((size_t)qcap * 2 * sizeof(uint32_t));
}

// The grid kernel's per-lane level counters are summed in kCntCopies copies
// (block b adds into copy b % kCntCopies, and every block sums the copies
// after the barrier): 304 blocks adding into one set of 512 words made the
// adds queue on a few cache lines.
constexpr uint32_t kCntCopies = 16;
constexpr uint32_t kCntParity = kCntCopies * 512;   // u32 per level parity

// A frontier word whose vertex has many out-arcs, queued so that every warp
// can take a share of its arcs.
struct HeavyEntry {
    unsigned long long F;   // live frontier lanes of the word
    uint32_t beg, deg;      // the vertex's arcs
    uint32_t g, pad;        // word group
};

// The prefilter's working memory (n entries an array; keep: n bits).
constexpr int kWalkLevels = 4;
struct Walks {
    uint32_t* c[kWalkLevels + 1];   // c[j][v]: walks of j arcs from v that never turn straight back (j >= 1)
    uint32_t* heavy;                // rows summed by whole blocks
    uint32_t* list[2];              // sources left, round by round
    uint32_t* keep;                 // which positions of the source list stay
    uint32_t* heavy_n;              // [kWalkLevels + 1]
    uint32_t* want;                 // the last c[j] there is (at least 2)
    uint32_t* probe;                // [3] zeroed: k_walk_probe's counts, blocks done
    uint32_t off;                   // no more than c[2]
    uint32_t max_deg;               // the graph's longest row
};

struct WaveParams {
    GraphDev g;
    uint32_t footnote;       // undirected: gamma~ uses deg(u)-1 for d >= 1
    uint32_t exhaustive;     // 1: no cut, write farness/reach of every source
    const uint32_t* sources; // the source queue: the degree order, or the deferred sources
    uint32_t* head;          // next position in `sources` (atomic)
    uint32_t n_end;          // sources are sources[*head .. n_end)
    TopK topk;
    unsigned long long* out_far;   // exhaustive outputs, indexed by vertex id
    uint32_t* out_reach;
    char* slot_base;         // CTA i: slot_base + i * slot_stride
    size_t slot_stride;
    // per-CTA slots: vertex tables of cta_entries entries (cta_entries = n
    // and tab_shift = 0: dense, vertex x is entry x; else hashed, cta_entries
    // = 2^(32 - tab_shift), and a wave making more than tab_limit entries is
    // given up and deferred)
    uint32_t cta_entries;
    uint32_t tab_shift;
    uint32_t tab_limit;
    // one-source-per-CTA kernel: entries of each vertex queue (a longer
    // frontier defers the source)
    uint32_t sparse_qcap;
    const uint32_t* lat_rows;   // k_lattice: the padded adjacency (launch_lattice_rows)
    const unsigned long long* lat_lb;   // k_lattice: per vertex, a lower bound on its farness (NULL: none)
    char* seed_base;         // the grid kernel's own slot (4 words per vertex)
    unsigned long long* stats;   // [ST_COUNT]
    int* err;
    unsigned long long lock_limit_ns;
    unsigned long long barrier_limit_ns;
    // grid-wide (seed / plain) kernels only
    GridBarrier* bar;
    uint32_t* gcnt;          // [2][kCntCopies][2][256] per-lane level counters (gamma, degree sum) by
                             // level parity, in copies that blocks add into by blockIdx % kCntCopies
    uint32_t* glist_n;       // [2] frontier list sizes
    uint32_t* glog_n;        // [1] cleared-word log size
    uint32_t* gchunk;        // [2] chunk counters of the frontier lists
    unsigned long long* garc; // [2] out-arcs of the frontier lists' words
    HeavyEntry* gheavy;      // heavy entries of the level being pushed
    uint32_t* gheavy_n;
    uint32_t gheavy_cap;
    uint32_t max_grid_waves;  // grid kernel: at most this many waves
    uint64_t heavy_words;   // grid kernel: a wave with fewer frontier words in total is light
    uint32_t pull_div;      // grid kernel: pull a level whose frontier words have >= n*W/pull_div out-arcs (0: never)
    uint32_t all_pull;      // grid kernel: pull every level after the first (a check of the pull path)
    // per-CTA kernel: a wave about to expand a level of at least defer_words
    // words, or of at least 8 * defer_words out-arcs, is given up and its
    // live sources appended to defer_src (0: never)
    uint32_t defer_words;
    uint32_t* defer_n;
    uint32_t* defer_src;
    // per-CTA kernel: each CTA stops after this many waves (0: when the queue is empty)
    uint32_t max_cta_waves;
    // when set, the sources end at *n_end_dev (read at launch)
    const uint32_t* n_end_dev;
    // optional trace: records of 4 u64 (layout in include/bcm.h, bcm_trace), NULL when off
    unsigned long long* trace;
    uint32_t trace_cap;      // records
    uint32_t* trace_n;       // records written (may exceed trace_cap; the excess is dropped)
    uint32_t trace_lanes;    // also record every lane's level state and end (needs trace)
    uint32_t nocut;          // top-k runs: never stop a source (every BFS runs to its end)
    // grid-wide kernel: the next wave's sources, picked by the leader block -- the next of the
    // queue, or (pick) the next that the walk bounds do not stop
    uint32_t* wave_src;      // [256]
    uint32_t* wave_n;
    uint32_t pick, undirected;
    uint32_t min_left;       // the launch ends once fewer sources than this are queued (0: never)
    uint32_t* walk_want;     // receives, when the launch ends, how many walk counts the prefilter wants
    Walks walks;
    uint32_t* light;         // grid-wide kernel: set when a narrow wave ended it; set on entry: nothing to do
    Threshold* snap;         // grid-wide and plain kernels: the threshold all blocks cut with (see store_snapshot)
};

// Trace record kinds (bits 60..63 of a record's second word).
enum TraceKind { TR_GRID_LEVEL = 0, TR_GRID_WAVE = 1, TR_CTA_WAVE = 2, TR_LANE_LEVEL = 3, TR_LANE_END = 4 };

// ---- preproc.cu
int launch_validate(const uint64_t* rp64, const uint32_t* col, uint32_t n, uint64_t m, int* err,
                    cudaStream_t s);
int launch_narrow_offsets(const uint64_t* rp64, uint32_t* rp32, uint32_t n, cudaStream_t s);
// *not_simple |= 1 unless every row is strictly increasing and free of its own vertex
// (scratch: simple_check_scratch_bytes(m))
size_t simple_check_scratch_bytes(uint64_t m);
int launch_simple_check(const uint32_t* rp32, const uint32_t* col, uint32_t n, uint64_t m, int* not_simple,
                        void* scratch, cudaStream_t s);
int launch_cc_reach(const uint32_t* rp, const uint32_t* col, uint32_t n, uint32_t max_degree, uint32_t* parent,
                    uint32_t* size, uint32_t* xlo, uint32_t* xhi, int* err, cudaStream_t s);
int launch_degree_order(const uint32_t* rp, uint32_t n, uint32_t* order, void* scratch,
                        size_t scratch_bytes, cudaStream_t s, uint32_t* max_degree = nullptr);
size_t degree_order_scratch_bytes(uint32_t n);
// stable LSD radix sort of (key, value) pairs on the low `bits` of the key
size_t radix_scratch_bytes(size_t count);
int radix_sort_pairs_u32(uint32_t* keys, uint32_t* vals, uint32_t* keys_tmp, uint32_t* vals_tmp,
                         size_t count, int bits, void* scratch, cudaStream_t s, bool* result_in_tmp);
int radix_sort_u64(uint64_t* keys, uint64_t* keys_tmp, size_t count, int bits, void* scratch,
                   cudaStream_t s, bool* result_in_tmp);
// exclusive scan of u32 counts into u32 offsets (out may alias in); returns total via *total_dev
size_t scan_scratch_bytes(size_t count);
int exclusive_scan_u32(const uint32_t* in, uint32_t* out, size_t count, uint32_t* total_dev,
                       void* scratch, cudaStream_t s);

// component labels: flags[v] = (parent[v] == v); parent[v] = rank[parent[v]]
int launch_root_flags(const uint32_t* parent, uint32_t n, uint32_t* flags, cudaStream_t s);
int launch_relabel(uint32_t* parent, const uint32_t* rank, uint32_t n, cudaStream_t s);

// ---- scc.cu
struct SccResult { uint32_t n_scc; };
size_t scc_scratch_bytes(uint32_t n, uint64_t m);
int launch_reverse_csr(const uint32_t* rp, const uint32_t* col, uint32_t n, uint64_t m, uint32_t* rrp,
                       uint32_t* rcol, void* scratch, size_t scratch_bytes, cudaStream_t s);
int launch_scc_bounds(const uint32_t* rp, const uint32_t* col, const uint32_t* rrp, const uint32_t* rcol,
                      uint32_t n, uint64_t m, uint32_t* comp, uint32_t* xlo, uint32_t* xhi, uint32_t* n_scc_host,
                      int refine, void* scratch, size_t scratch_bytes, int* err, cudaStream_t s);

// ---- msbfs.cu
int launch_grid_waves(const WaveParams& p, int W, int blocks, int threads, cudaStream_t s);
int launch_cta_waves(const WaveParams& p, int W, int blocks, int threads, cudaStream_t s);
// c[1] and c[2] (K.heavy: n entries of scratch, K.heavy_n: kWalkLevels + 1)
int launch_walk_base(const uint32_t* rp, const uint32_t* col, uint32_t n, const Walks& K, bool undirected,
                     cudaStream_t s);
// Stopping rule at levels 0 and 1 and walk bounds for the sources p.sources[*p.head .. end) of a simple
// graph; those it cannot stop go to out in the same order, their count to *out_n (device memory).
int launch_prefilter(const WaveParams& p, const Walks& K, bool undirected, uint32_t* out, uint32_t* out_n,
                     cudaStream_t s);
// the same for p's sources with the counts already there, against the threshold by now
int launch_refilter(const WaveParams& p, const Walks& K, bool undirected, uint32_t* out, uint32_t* out_n,
                    cudaStream_t s);
int launch_plain_source(const WaveParams& p, uint32_t it, uint32_t* stamp, uint32_t* lists,
                        int blocks, int threads, cudaStream_t s);

int max_coop_blocks(int kind, int W, int threads);   // kind 0 grid waves, 1 plain
int cta_blocks_per_sm(int W, int threads);
// one source per CTA (high-diameter graphs): sources p.sources[*p.head .. n_end)
int launch_sparse(const WaveParams& p, int blocks, int threads, cudaStream_t s);
int sparse_blocks_per_sm(int threads);

// ---- lattice.cu: one source per CTA on a padded adjacency of rw = 4 or 8 entries per vertex
// (undirected graphs of largest degree <= rw, n <= 2^28)
int launch_lattice_rows(const uint32_t* rp, const uint32_t* col, uint32_t n, int rw, uint32_t* rows, cudaStream_t s);
int launch_lattice(const WaveParams& p, int rw, int blocks, int threads, cudaStream_t s);
int lattice_threads(uint32_t n);
int lattice_blocks_per_sm(uint32_t n, int threads, int rw);
bool lattice_smem(uint32_t n);   // its visited bitmap lies in shared memory
size_t lattice_slot_bytes(uint32_t n, uint32_t qcap);
// Landmark bounds for k_lattice's sources (landmark.cu).  Working memory, carved out of one block of
// landmark_bytes(n):
struct Landmarks {
    float4* dist;                    // [n] distances from the four landmarks (all ones: not in their component)
    uint32_t* mind;                  // [n] distance to the nearest landmark so far
    uint32_t* lv_cnt;                // [4][n + 1] vertices within a distance of landmark i
    unsigned long long* lv_sum;      // [4][n + 1] their distance sum
    uint32_t* queue;                 // [2][n] BFS queues past the part in shared memory
    uint32_t* bitmap;                // [n bits] where shared memory is too small
    unsigned long long* lb;          // [n] the best bound on f(v) known
    unsigned long long* joint;       // [n] the joint bound (k_lm_joint)
    unsigned long long* sample;      // [kLmSample] the joint bound of sampled sources
    uint32_t *key, *key_tmp, *val, *val_tmp;   // [n] sources by bound
    uint32_t *list_a, *list_b;       // [n] sources left after the one-landmark / the joint bound
    void* radix;
    struct Info {
        uint32_t size, valid;        // of the landmarks' component; 0: distances too large, no bound
        uint32_t levels[4];
        uint32_t n_a, n_b, go;       // list lengths; the joint bound is worth taking
    }* info;
};
size_t landmark_bytes(uint32_t n);
Landmarks landmark_carve(void* base, uint32_t n);
// distances and one-landmark bounds; *order gets the n_src sources p.sources[0..) by ascending bound
int launch_landmarks(const WaveParams& p, const Landmarks& L, int rw, uint32_t n_src, uint32_t** order, cudaStream_t s);
// sources order[first..n_src) that no bound stops -> L.list_b, their count in L.info->n_b; the others
// are counted as cut
int launch_landmark_filter(const WaveParams& p, const Landmarks& L, const uint32_t* order, uint32_t first,
                           uint32_t n_src, cudaStream_t s);

// ---- allpairs.cu: farness and reach of every vertex, the lanes of a wave being targets
struct AllPairs {
    uint32_t n;
    const uint32_t *rp, *col;      // out-arcs, rows by degree descending (launch_sorted_rows) ...
    const uint32_t* vertex;        // ... row i that of vertex[i]; NULL: row i is vertex i, in any order
    const uint32_t* pos;           // the row of each vertex
    const uint32_t* grp;           // the graph's own offsets
    const uint32_t *rrp, *rcol;    // its in-arcs (NULL: not there)
    char* slots;                   // one per cluster, allpairs_slot_bytes apart
    size_t slot_stride;
    uint32_t* lanes;               // [clusters][48]
    unsigned long long* far;       // [n] zeroed
    uint32_t* reach;               // [n] zeroed
    unsigned long long* stats;     // [ST_COUNT]
    // where another kernel can take over: what the waves have cost so far, and how many rounds of
    // waves of 64 sources that kernel would run (NULL: there is none)
    struct Pace {
        unsigned long long ns, levels, found;   // of the levels looked at: time, their number, (row, lane) pairs gained
        uint32_t looks, quit;                   // quit: given up, far and reach are not complete
    }* pace;
    uint32_t rival_rounds;
    uint32_t wave_step;            // with pace: wave i takes the targets of wave i * wave_step mod the waves (coprime)
};
constexpr size_t kAllPairsL2 = 130ull << 20;   // (R-MAT 2^16: 129 MB at 256 lanes 12.2 ms, 70 MB at 128 13.9)
constexpr uint32_t kAllPairsTopkN = 16384;
size_t sorted_rows_bytes(uint32_t n, uint64_t m);
size_t sorted_rows_scratch_bytes(uint32_t n);
int launch_sorted_rows(const uint32_t* grp, const uint32_t* gcol, const uint32_t* order, uint32_t n, uint64_t m,
                       void* rows, void* scratch, cudaStream_t s);
void sorted_rows_use(AllPairs* a, const void* rows, uint64_t m, const uint32_t* order);
int launch_allpairs(const AllPairs& p, int W, int C, int clusters, cudaStream_t s);
// the top-k from every vertex's farness and reach (rank: [n] zeroed)
int launch_rank_topk(const unsigned long long* far, const uint32_t* reach, uint32_t n, uint32_t* rank, const TopK& T,
                     cudaStream_t s);

// launch bookkeeping (api.cu)
void note_launch(int count = 1);
// sets the calling thread's bcm_last_error() message (api.cu)
void set_error_message(const char* msg);

}  // namespace bcm
