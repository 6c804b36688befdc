// Internal declarations shared by the kernels and the host runtime of the
// hybrid-transfer graph engine.  Nothing here is part of the public C ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace hytg {

constexpr int kRoutes = 5;            // NONE, CACHE, F, C, Z (hytg_route)
constexpr int kRouteNone = 0, kRouteCache = 1, kRouteF = 2, kRouteC = 3, kRouteZ = 4;

// Frontier bitmap: one bit per vertex, 32-bit words, padded to a multiple of
// 32 words; the planning kernels walk it in units of four words (plan.cu).  One
// bitmap serves a whole run: k_bin clears the bits it takes, the relax
// kernels set the bits of changed vertices for the next iteration.
constexpr int kBitmapPadWords = 32;

// Route edges per entry of the tile index (the list entry that owns the tile's
// first edge) and at most per run, the unit of work of a warp of the relax kernels.
constexpr int kRelaxBlock = 256;
constexpr int kTile = 2048;
constexpr int kRunShift = 8, kRun = 1 << kRunShift;

// The compaction buffer is a multiple of this many edges.
constexpr int kCompactUnit = 2048;

constexpr int kSelectBlock = 512;    // 128 registers per thread: the per-route sums stay in registers

enum Algo : int { kBFS = 0, kSSSP = 1, kCC = 2, kPR = 3, kPPR = 4 };

// Cost-model parameters of one iteration (Sec. V-A).  alpha, beta, gamma are
// rationals num / 1e6 so that the device decision is exact.
struct CostParams {
    unsigned long long alpha_num, beta_num, gamma_num;   // over kParamDen
    unsigned long long m, MR;
    unsigned long long d1;          // bytes read per edge (4 or 8)
    unsigned long long d2;          // bytes per index entry (8)
    unsigned int n_cached;          // partitions [0, n_cached) are resident
    int force_route;                // -1 cost model; 1..4 forced route; 5 random
    unsigned long long seed;        // for force_route 5
    unsigned int iteration;
};
constexpr unsigned long long kParamDen = 1000000ull;

// Device-side summary of one iteration, copied to the host in one piece
// together with the per-partition arrays that follow it in memory.
struct alignas(16) Summary {
    unsigned long long n_active;                 // active vertices (any degree)
    unsigned long long route_entries[kRoutes];   // list entries (active, degree > 0)
    unsigned long long route_edges[kRoutes];     // active edges
    unsigned long long route_lines[kRoutes];     // 128-byte lines (cost-model count)
    unsigned long long route_entry_base[kRoutes];// first index of each route in the list
    unsigned long long route_tile_base[kRoutes]; // first tile of each route
    unsigned int route_parts[kRoutes];
    unsigned int pending_min;                    // bucketed SSSP: smallest pending dist
    unsigned long long pending;                  // bucketed SSSP: active but not yet eligible
    unsigned long long alive;                    // batched: sources with a frontier this iteration
};

// Per-partition arrays, laid out right after the Summary in one buffer.
struct PartArrays {
    unsigned long long *n_act;      // |A_i|
    unsigned long long *entries;    // active vertices with degree > 0
    unsigned long long *edges;      // sum of D_o over A_i
    unsigned long long *lines;      // 128-byte lines spanned (all arrays read)
    unsigned long long *route_entry;// first list index of the partition inside its route
    unsigned long long *route_edge; // first edge index of the partition inside its route
    unsigned long long *cursor;     // fill cursor: entries (low 24 bits) | edges << 24
    unsigned long long *pending;    // bucketed SSSP: pending vertex count
    unsigned long long *pending_inv;// bucketed SSSP: max of ~dist over pending vertices
    unsigned long long *prio;       // delta-first order: sum over A_i of |delta| * 2^24 (PageRank)
    unsigned char *route;           // hytg_route
    const unsigned long long *alive;// batched: source mask of the frontier (or nullptr)
};

// The list of active vertices of one iteration, grouped by route and, inside
// a route, ordered by partition and vertex id.
struct ListArrays {
    unsigned long long *ebase;      // first edge of the entry in its route's edge space
    unsigned long long *soff;       // row offset of the vertex (its first edge in the CSR)
    unsigned int *pay;              // value pushed along its edges (uint32 or float bits)
    unsigned int *tile_first;       // per route tile: list entry (route-relative) holding its first edge
    unsigned long long cap_entries; // capacity of ebase / soff / pay
    unsigned long long cap_tiles;   // capacity of tile_first
    unsigned int *err;              // device word: nonzero if an index check failed
    unsigned long long *pay64;      // batched runs: per-source frontier word of the entry
    unsigned int *vid;              // batched runs: the entry's vertex
};

// ------------------------------------------------------------------ helpers
__device__ __forceinline__ unsigned long long lines_spanned(unsigned long long start,
                                                            unsigned long long len,
                                                            unsigned long long m) {
    return len == 0 ? 0ull : (start + len - 1) / m - start / m + 1;
}

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// inclusive warp scan
__device__ __forceinline__ unsigned long long warp_scan_u64(unsigned long long x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// Counter-based mix used only for the "random route" test mode.
__host__ __device__ __forceinline__ unsigned long long mix64(unsigned long long x) {
    x ^= x >> 33; x *= 0xff51afd7ed558ccdull;
    x ^= x >> 33; x *= 0xc4ceb9fe1a85ec53ull;
    x ^= x >> 33;
    return x;
}

// ------------------------------------------------------------- launchers
// Streaming multiprocessors of the current device (cudaDevAttrMultiProcessorCount),
// read once per device and cached; grid caps are multiples of it.
unsigned int device_sms();

struct GraphDev {
    const unsigned long long *off;      // V+1 row offsets (device)
    unsigned long long V, n_words_alloc;
    const unsigned int *part_wb;        // partition bounds in bitmap words, N+1
    const unsigned long long *part_eb;  // partition bounds in edges, N+1
    const unsigned int *round_part;     // partition holding word 32 * r, per 32-word round
    unsigned int N;
};

// Control block of the device-driven iteration loop (a CUDA graph whose
// WHILE node repeats plan + cache/Z relax until an iteration needs the F or C
// route, the frontier is empty, or the iteration cap is reached).
enum LoopStatus : unsigned int { kLoopRun = 0, kLoopDone = 1, kLoopHost = 2, kLoopMaxIt = 3, kLoopCancel = 4 };
struct LoopCtl {
    unsigned int status;            // LoopStatus when the loop exits
    unsigned int it;                // number of the iteration being planned
    unsigned int bucket;            // SSSP delta-stepping bucket limit (~0u: off)
    unsigned int work;              // 1: this iteration's bin and relax run on the device
    unsigned int n_rec, rec_cap;    // iteration records written / capacity
    unsigned long long delta;       // bucket width (0: no buckets)
    unsigned long long max_it;
    unsigned long long m;           // request bytes (link bytes of zero-copy lines)
    void *rec;                      // hytg_iter_record[rec_cap]
    // F and C iterations inside the loop ("device_loop" 2): the IF-node
    // handle of every partition's F task (nullptr: F iterations go to the
    // host) and of the C route (0: C iterations go to the host)
    const unsigned long long *f_handles;
    unsigned long long c_handle;
    unsigned long long c_cap;       // compaction buffer, in edges (larger C routes go to the host)
    const unsigned char *route;     // per-partition routes of the iteration
    const unsigned long long *part_eb;
    unsigned int n_parts, dst_bits, w_bits;   // w_bits 0: the run reads no weights
    // a word of mapped host memory that the host sets to end the loop at the
    // next iteration boundary (a run past its deadline); nullptr: none
    const volatile unsigned int *cancel;
    // totals over the device iterations of this launch
    unsigned long long route_parts[kRoutes], route_entries[kRoutes], route_edges[kRoutes];
    unsigned long long z_lines, vertices, edges, iterations;
    unsigned long long f_parts, f_bytes, c_iters, c_lines;
    // small-frontier iterations (k_tail): allowed in this graph, chosen for the
    // iteration being planned, the first iteration it may take after one that
    // it refused, iterations it has run; body runs (each launches the whole body)
    unsigned int tail_ok, tail_gather, tail, tail_not;
    unsigned long long tail_its, bodies;
};

// Small-frontier iterations: queue entries (a thread each), partitions whose
// routes one block decides, and the frontier that k_select hands over.  A
// 1021 x 1031 mesh (CC, device time): frontiers up to 2,048 vertices 26.2 ms,
// up to the whole queue 19.3 ms; more edges than 4 a thread gain nothing on
// meshes and make R-MAT frontiers (a few lists of thousands of edges) try in
// vain.
constexpr unsigned int kTailQueue = 4096, kTailParts = 1024, kTailActive = 4096, kTailEdges = 16384;
enum TailExit : int { kTailAgain = 0, kTailDone = 1, kTailMaxIt = 2, kTailCancel = 3 };

struct AlgoState {
    int algo;
    unsigned int *val;       // BFS level / SSSP dist / CC label
    float *rank, *delta;     // PageRank state
    float *rank_lo;          // what rank's roundings left out (rank_add)
    float damping, eps;
    unsigned int *bm_cur, *bm_next;
    unsigned int *overflow;  // device flag
    unsigned int n_arrays;   // edge arrays read per edge (1 or 2)
    const unsigned int *perm;// internal id -> original id (hub sorting), or nullptr
    // PageRank pushes to hub ids [0, n_hub_rep) go to replica rows of n_hub_rep sums:
    // a plain relax adds each to its SM's row (smid % kHubReplicas), k_relax_rank
    // its blocks' sums to the first kRankRows; all rows join delta once per
    // iteration, those first ones also when a second pass looks at their ids
    float *hub_rep;
    unsigned int n_hub_rep;
    unsigned int bucket_limit;  // SSSP delta-stepping: only dist < limit is eligible (~0u: off)
    LoopCtl *loop;              // device loop: bucket from loop->bucket; bin/relax run if loop->work
    int prio;                   // PageRank/PPR: k_count sums |delta| per partition (delta-first order)
    // batched runs (BatchMode): k_bin takes the per-source frontier word as payload
    int batch_mode;
    const unsigned long long *b_fr;   // BFS/SSSP: 64-bit source mask per vertex
    const unsigned int *b_fr32;       // PPR: 32-bit seed mask per vertex
    unsigned long long *src_work;     // sum over entries of popcount(mask) * degree
    unsigned long long V;
};
// rank[v] += dl, where rank and its low part hold hi and lo.  A rank is the sum of
// a hundred or two takes, and their roundings were the largest part of the
// result's error (R-MAT 20, resident: 2.2e-7 in the 2-norm), more so since a
// second pass takes hubs too; the exact error of each sum (Knuth's two-sum) is kept
// beside it (0.5e-7; the resident run 2 % longer).
__device__ __forceinline__ void rank_add(const AlgoState &st, unsigned long long v, float hi, float lo, float dl) {
    const float s = hi + dl, b = s - hi;
    st.rank[v] = s;
    st.rank_lo[v] = lo + ((hi - (s - b)) + (dl - b));
}
// Edges from which a PageRank relax sums hub ids in shared memory (rank_ids).
constexpr unsigned long long kRankNarrow = 1ull << 14, kRankWide = 1ull << 23;

enum BatchMode : int { kBatchNone = 0, kBatchBFS = 1, kBatchSSSP = 2, kBatchPPR = 3 };

// Per-source state of batched runs and serving lives in frames of
// kFrameSources consecutive sources, so that serving can allocate and release
// it eight queries at a time.  Frame g holds sources [8 g, 8 g + 8): BFS/SSSP
// val[g][v * 8 + (s & 7)] (V * 32 bytes); PPR delta[g], rank[g], msg[g], each
// V * 8 floats (V * 96 bytes in all).  A warp that reads every source of one
// vertex reads one 32-byte sector per frame, as a contiguous vertex-major
// layout would.  Only frames of sources that can be active are read.
constexpr unsigned int kFrameSources = 8;
constexpr unsigned int kMaxFrames = 8;           // 64 BFS/SSSP sources; PPR uses 4 (32 seeds)
constexpr unsigned int kMaxPprFrames = 4;
struct BatchState {
    int mode;
    unsigned long long *fr, *vis, *nxt;   // BFS/SSSP source masks
    unsigned int *val[kMaxFrames];        // BFS level / SSSP distance frames (nullptr: none)
    float *delta[kMaxPprFrames], *rank[kMaxPprFrames], *msg[kMaxPprFrames];   // PPR frames
    unsigned int *fr32;                   // PPR seeds taken at v this iteration
    float *hub;                           // PPR pushes to ids [0, n_hub): kBatchHubCopies copies of
    unsigned int n_hub;                   // n_hub rows of kMaxPprSeeds floats (b_hub)
    unsigned long long *alive;            // OR of every vertex's frontier mask (serving)
    const LoopCtl *loop;                  // device loop: level from loop->it; relax gated by loop->work
    unsigned int sparse_below;            // SSSP/PPR relax: a warp whose 32 edges carry fewer than
                                          // this many active sources per edge on average loops
                                          // over sources per lane (0: never)
};
__device__ __forceinline__ unsigned int *bval(const BatchState &b, unsigned long long v, unsigned int s) {
    return b.val[s >> 3] + v * kFrameSources + (s & 7);
}
__device__ __forceinline__ float *bdelta(const BatchState &b, unsigned long long v, unsigned int s) {
    return b.delta[s >> 3] + v * kFrameSources + (s & 7);
}
__device__ __forceinline__ float *brank(const BatchState &b, unsigned long long v, unsigned int s) {
    return b.rank[s >> 3] + v * kFrameSources + (s & 7);
}
__device__ __forceinline__ float *bmsg(const BatchState &b, unsigned long long v, unsigned int s) {
    return b.msg[s >> 3] + v * kFrameSources + (s & 7);
}
constexpr unsigned int kHubReplicas = 256;
// The first of them also take the block sums of k_relax_rank, in turn.
constexpr int kRankRows = 8;
// Batched PPR's hub copies, in the memory of the single-source replicas.
constexpr unsigned int kBatchHubIds = 64, kBatchHubCopies = 16, kMaxPprSeeds = kMaxPprFrames * kFrameSources;
__device__ __forceinline__ float *b_hub(const BatchState &b, unsigned int copy, unsigned int v, unsigned int s) {
    return b.hub + ((size_t)copy * b.n_hub + v) * kMaxPprSeeds + s;
}

// log2 of a power of two, else -1.
inline int log2_exact(unsigned long long m) {
    if (m == 0 || (m & (m - 1))) return -1;
    int s = 0;
    while ((1ull << s) < m) ++s;
    return s;
}
cudaError_t launch_count(const GraphDev &g, const AlgoState &st, const PartArrays &pa,
                         unsigned long long m, cudaStream_t s);
// With ctl, the device loop's decision too: cond is the WHILE node's condition.
cudaError_t launch_select(const GraphDev &g, const PartArrays &pa, const CostParams &cp,
                          Summary *sum, cudaStream_t s, LoopCtl *ctl = nullptr,
                          unsigned long long cond = 0);
cudaError_t launch_bin(const GraphDev &g, const AlgoState &st, const PartArrays &pa,
                       const ListArrays &la, const Summary *sum, cudaStream_t s);

// Edge source of a relax / gather launch.
enum EdgeMode : int { kModeHost = 0, kModeDevice = 1, kModeCompact = 2 };

// The edge arrays a task reads, in host memory or copied to the device.  The
// CSR arrays are bit-packed at load: entry e takes `bits` bits, from bit
// e * bits - off of the array (least significant bit first), so any run of
// edges is a run of words that can be copied or read as it is.  Targets take
// ceil(log2 V) bits and weights those of the largest one: on R-MAT 24 with
// weights up to 64, 24 and 7 bits of 32 each, so the host link, the staging
// slots and the cache move or hold 1.3x (BFS, CC, PageRank) to 2.1x (SSSP)
// more edges per byte.  Such runs are bound by the link: at a budget of 25 %
// of the graph (R-MAT 24, device time) BFS went from 6.0 to 3.9 ms, SSSP from
// 22.8 to 10.7 ms, PPR from 278 to 229 ms (46 -> 24 GB copied).  Entries keep
// a fixed width rather than gaps of sorted rows, so any edge of any row order
// is found by its index alone.  The compaction buffer holds plain words.
struct EdgeSrc {
    const unsigned int *dst, *w;        // targets; weights or nullptr
    unsigned int dst_bits, w_bits;
    long long dst_off, w_off;
    unsigned long long e_lo, e_hi;      // edges present: [e_lo, e_hi)
};

// The words to copy for entries [e0, e0 + n) of `bits` bits: from the 16-byte
// boundary at or below the first entry to the word of the last one.
struct WordSpan {
    unsigned long long w0, n;
};
__host__ __device__ inline WordSpan word_span(unsigned long long e0, unsigned long long n, unsigned int bits) {
    const unsigned long long w0 = (e0 * bits / 32) & ~3ull;
    return {w0, n ? ((e0 + n) * bits + 31) / 32 - w0 : 0};
}

struct RelaxTask {
    int route;                          // which route's list / tiles
    int mode;                           // EdgeMode: in a compacted buffer an edge is its place in the route
    EdgeSrc src;
    unsigned long long k_begin, k_end;  // edge range in the route's edge space
    unsigned long long first_entry;     // route-relative entry holding k_begin
    bool device_sized;                  // take k_end from the summary (k_begin = 0)
    unsigned long long *link_ctr;       // host-memory reads (Z relax, C gather): {32-byte
                                        // sectors, 128-byte lines} read, or nullptr
    // One partition's F task inside the device loop: its first edge in the F
    // route's edge space, its active edges and its first list entry, read on
    // the device where k_select and k_bin left them (nullptr: host bounds)
    const unsigned long long *dev_edge, *dev_len, *dev_entry;
    // A second pass's push: its list is [sp_rbase, ...) of the second-pass
    // arrays, sized by the range's cursor (nullptr: a route's list)
    const unsigned long long *sp_cursor;
    unsigned long long sp_rbase, sp_tbase;
    // The cursor of the second pass that follows this launch, cleared by it
    unsigned long long *sp_reset;
};

// Cursor of a second pass's list: entries in the low 30 bits, edges above.
constexpr unsigned long long kSpEntries = (1ull << 30) - 1, kSpEdgesMax = (1ull << 34) - 1;

struct TailArgs {
    GraphDev g;
    AlgoState st;
    EdgeSrc cache, host;
    CostParams cp;
    unsigned long long m;               // request bytes
    int m_shift;                        // log2 of m when it is a power of two, else -1
    int gather;                         // 1: the compaction route runs here too
    LoopCtl *ctl;
    unsigned int *queue[2];             // kTailQueue vertices each
    unsigned long long *link_ctr;       // per route {sectors, lines}
    unsigned int *err;
    unsigned long long cond;            // the WHILE node's condition
};
cudaError_t launch_tail(const TailArgs &a, cudaStream_t s);

cudaError_t launch_relax(const AlgoState &st, const ListArrays &la, const Summary *sum,
                         const RelaxTask &t, int grid_cap, cudaStream_t s);
// Both tasks device-sized (routes of the current list); plain runs only.
cudaError_t launch_relax_pair(const AlgoState &st, const ListArrays &la, const Summary *sum,
                              const RelaxTask &ta, const RelaxTask &tb, int grid, cudaStream_t s);
// Second pass (Sec. VI-A) over vertices [vlo, vhi) (vlo a multiple of 32)
// whose edges [E0, E1) are resident in src:
// a take launch, which lists the vertices it takes as k_bin lists a route's,
// and a relax over that list.  The list's entries lie at [vlo, vhi) and its
// tiles from `tbase` of arrays shared by every second pass of a run, whose
// ranges never overlap; *cursor must be zero (see RelaxTask::sp_reset).
struct SecondPassRange {
    unsigned long long vlo, vhi, E0, E1;
    unsigned long long tbase;            // first tile of the range's slice
    unsigned long long *cursor;          // packed entries and edges of its list
    unsigned long long *edges_out;       // statistics: edges taken
    EdgeSrc src;
};
cudaError_t launch_second_pass(const AlgoState &st, const unsigned long long *off, const SecondPassRange &r,
                               const ListArrays &la, const Summary *sum, cudaStream_t s);
// Batched PPR: the second pass over a resident range, taking each seed whose
// residual rose above eps again (K seeds).
cudaError_t launch_second_pass_batched(const BatchState &b, const unsigned long long *off,
                                       const SecondPassRange &r, const ListArrays &la, const Summary *sum,
                                       unsigned int K, float damping, float eps, unsigned int *bm,
                                       cudaStream_t s);
cudaError_t launch_gather(const ListArrays &la, const Summary *sum, const RelaxTask &t,
                          unsigned int *out_dst, unsigned int *out_w, int grid_cap,
                          cudaStream_t s, const LoopCtl *loop = nullptr);

cudaError_t launch_b_init(const BatchState &b, unsigned long long V, unsigned long long n_words_alloc,
                          const unsigned int *src_dev, unsigned int K, float base, unsigned int *bm,
                          cudaStream_t s);
// Fill frame g of the batched state with "no value" (BFS/SSSP: unreached;
// PPR: zero delta and rank), as every frame must hold before it is used.
cudaError_t launch_frame_init(const BatchState &b, unsigned long long V, unsigned int g, cudaStream_t s);
cudaError_t launch_b_commit(const BatchState &b, unsigned long long V, unsigned long long n_words_alloc,
                            unsigned int level, unsigned int *bm, cudaStream_t s);
cudaError_t launch_b_take(const BatchState &b, const unsigned long long *off,
                          unsigned long long n_words_alloc, unsigned int K, float damping, float eps,
                          unsigned int *bm, cudaStream_t s);
cudaError_t launch_relax_batched(const BatchState &b, const ListArrays &la, const Summary *sum,
                                 const RelaxTask &t, int grid_cap, unsigned int *bm,
                                 unsigned int *overflow, cudaStream_t s);
cudaError_t launch_serve_admit(const BatchState &b, unsigned long long V, unsigned int slot,
                               unsigned int src, float base, unsigned int *bm, cudaStream_t s);
cudaError_t launch_serve_extract(const BatchState &b, unsigned long long V, unsigned int slot,
                                 const unsigned int *perm, unsigned int offset, void *out,
                                 double *sums, cudaStream_t s);
cudaError_t launch_b_finalize(const BatchState &b, unsigned long long V, unsigned int K,
                              const unsigned int *perm, void *out, double *sums, cudaStream_t s);

cudaError_t launch_zero_u64(unsigned long long *p, unsigned long long n, cudaStream_t s);
// Copy n 4-byte words from mapped host memory to device memory with 16-byte
// loads (the device loop's F copy where a memcpy node cannot be used);
// gated by loop->work.  Both addresses 16-byte aligned, n a multiple of 4
// except for the tail, which is copied word by word.
cudaError_t launch_copy_words(const unsigned int *src, unsigned int *dst, unsigned long long n,
                              const LoopCtl *loop, cudaStream_t s);
cudaError_t launch_init(const AlgoState &st, unsigned long long V, unsigned long long n_words_alloc,
                        unsigned int source, cudaStream_t s);
cudaError_t launch_pr_finalize(const AlgoState &st, unsigned long long V, float *out,
                               double *sums, cudaStream_t s);
cudaError_t launch_pr_frontier(const AlgoState &st, unsigned long long V,
                               unsigned long long n_words_alloc, cudaStream_t s);
cudaError_t launch_hub_reduce(const AlgoState &st, cudaStream_t s);
cudaError_t launch_cc_jump(const AlgoState &st, unsigned long long n_words_alloc, cudaStream_t s);
cudaError_t launch_cc_final(const AlgoState &st, unsigned long long V, unsigned int *tmp,
                            unsigned int *out, cudaStream_t s);
cudaError_t launch_pr_rank(const AlgoState &st, unsigned long long V, float *out, cudaStream_t s);
cudaError_t launch_to_original(const unsigned int *perm, const unsigned int *in, float *out,
                               unsigned long long V, cudaStream_t s);
cudaError_t launch_upload_bitmap(const unsigned char *active_dev, unsigned int *bm,
                                 unsigned long long V, unsigned long long n_words_alloc,
                                 cudaStream_t s);
cudaError_t launch_red_probe(unsigned int *idx, float *d, unsigned long long n, int skew, bool gen,
                             cudaStream_t s, float *rep = nullptr, unsigned int n_rep = 0);
cudaError_t launch_frame_probe(const unsigned int *idx, float *d, unsigned long long n, int width,
                               cudaStream_t s);
cudaError_t launch_stage_copy(const unsigned int *src, unsigned int *dst, unsigned long long n,
                              unsigned int blocks_per_sm, cudaStream_t s);
cudaError_t launch_zc_probe(const uint4 *src, unsigned long long n16, unsigned long long *sink,
                            int grid, cudaStream_t s);

}  // namespace hytg
