// Push relax kernels over the active edges of one route (Sec. II-A push
// model; Sec. VI-C processing kernels), and the compaction gather of the C
// route (Sec. II-B ExpTM-compaction, here done by the GPU over the host link).
//
// The walk over a route's active edges (a warp per run of up to 256 of them) is in
// edge_runs.cuh; a warp's loads cover consecutive edges of the same or
// adjacent lists: 128-byte lines when the lists are long, and neighbouring
// lists share lines when consecutive vertices are active.
//
// Edge sources (the route's transfer method; packed as EdgeSrc says):
//   host    zero-copy loads from pinned, device-mapped host memory (Eq. 3 route);
//   device  a device copy of a run of edges (cache and F routes);
//   compact the compaction buffer: plain words in route order.
#include "common.cuh"
#include "edge_runs.cuh"

namespace hytg {

namespace {

// cur: v's value, read shortly before (BFS, SSSP, CC); hub_rep: this SM's
// replica row of the hub accumulators (PageRank only: launches with too few edges
// for k_relax_rank, and the zero-copy route's).
template <int ALGO>
__device__ __forceinline__ void relax_edge(const AlgoState &st, unsigned int v, unsigned int pay,
                                           unsigned int w, unsigned int cur, float *hub_rep) {
    if (ALGO == kPR || ALGO == kPPR) {
        // fire-and-forget reduction; the next frontier is rebuilt from delta
        // (delta > eps) by k_pr_frontier once every relax of the iteration is
        // done.  Pushes to the hottest vertices (hub-sorted ids below
        // n_hub_rep) go to this SM's replica, so that the SMs' updates do not
        // serialise on one L2 address.
        if (v < st.n_hub_rep) atomicAdd(&hub_rep[v], __uint_as_float(pay));
        else atomicAdd(&st.delta[v], __uint_as_float(pay));
    } else {
        unsigned int nv;
        if (ALGO == kBFS) {
            nv = pay + 1u;
        } else if (ALGO == kSSSP) {
            const unsigned long long s = (unsigned long long)pay + w;
            if (s >= 0xFFFFFFFEull) { *st.overflow = 1u; return; }
            nv = (unsigned int)s;
        } else {
            nv = pay;
        }
        // Fire-and-forget min and frontier bit when the pushed value beats the
        // value seen now.  If a concurrent push lowered v further in between,
        // v is still marked active: it then re-pushes its (current) value
        // next iteration, which is redundant but never wrong for min-updates.
        if (nv < cur) {
            atomicMin(&st.val[v], nv);
            atomicOr(&st.bm_next[v >> 5], 1u << (v & 31));
        }
    }
}

// Edges whose loads one lane keeps in flight: four runs through the walk's
// steps, then four target loads, then (BFS, SSSP, CC) four value loads, then
// the reductions.
constexpr int kSteps = 4;

// The lane's edges of one step group: targets and weights, then the pushes.
template <int ALGO>
__device__ __forceinline__ void relax_edges(const AlgoState &st, const RelaxTask &t,
                                            const Edge<false> (&ed)[kSteps], float *hub_rep) {
    constexpr bool rank = ALGO == kPR || ALGO == kPPR;
    unsigned int dv[kSteps], wv[kSteps] = {}, cur[kSteps];
    load_entries<false>(t.src.dst, t.src.dst_bits, ed, dv);
    if (ALGO == kSSSP) load_entries<true>(t.src.w, t.src.w_bits, ed, wv);
    if (!rank) {
        // the values are read together before any reduction is issued (a
        // reduction between them would make the loads wait for one another)
#pragma unroll
        for (int q = 0; q < kSteps; ++q) cur[q] = ed[q].ok ? __ldcg(&st.val[dv[q]]) : 0u;
    }
#pragma unroll
    for (int q = 0; q < kSteps; ++q)
        if (ed[q].ok) relax_edge<ALGO>(st, dv[q], ed[q].pay, wv[q], rank ? 0u : cur[q], hub_rep);
}

template <int ALGO>
__global__ void __launch_bounds__(kRelaxBlock, 3) k_relax(AlgoState st, ListArrays la,
                                                       const Summary *sum, RelaxTask t) {
    if (st.loop && !st.loop->work) return;
    unsigned long long kb, ke;
    const RouteView rv = task_view(t, sum, kb, ke);
    float *hub_rep = st.hub_rep ? st.hub_rep + (size_t)(sm_id() % kHubReplicas) * st.n_hub_rep : nullptr;
    LinkCount lc;
    walk_task<kSteps, false, ALGO == kSSSP>(la, rv, t, kb, ke, lc, [&](const Edge<false> (&ed)[kSteps], unsigned long long) {
        relax_edges<ALGO>(st, t, ed, hub_rep);
    });
    flush_link(lc, t.link_ctr);
}

// PageRank and PPR pushes with the hottest targets summed on chip.  What bounds
// these relaxes is the rate of L2 reductions: 190 G/s to spread-out addresses,
// 140 to 165 with R-MAT's in-degree skew and per-SM replicas of 4,096 hub ids.
// Hub sorting puts the hottest targets at the lowest ids, so a block of 1,024
// threads (one per SM) sums the pushes to ids below ns in shared memory and adds
// the sums to memory at its end, four ids per vector reduction; a probe with the
// skew of 2^20 / 2^24 vertices then runs at 261 / 221 G pushes/s (ns = 16,384)
// against 137 / 166 with the replicas, and the relax of R-MAT 24's cache, 157 M
// edges, at 240 G pushes/s against 94.  The sums go to kRankRows rows of the hub
// replicas in turn (ids beyond the replicas: to delta), which a second pass adds
// to the residuals that it looks at (k_sp_take), as the end of the iteration adds
// all replicas: R-MAT 20, resident, 71 iterations instead of 97.  Whole runs:
// 22.5 -> 16 ms there, PPR on R-MAT 24 238 -> 210 ms.  The rows are for the
// rounding: with F tasks and their second passes an iteration has tens of
// launches, each of 152 or 304 blocks, and thousands of additions to one running
// 32-bit sum per hub doubled the result's error (PageRank, R-MAT 19 in 32
// partitions at a budget of 30 %: 1.9e-7 with the replicas, 4.6e-7 with sums into
// delta, 2.7e-7 with eight rows; with rank_add's low parts 0.8e-7).  TB: a second,
// device-sized task in the same launch.
//
// The kRankHot hottest ids have a sum per lane: an addition to shared memory is
// a compare-and-swap loop, and where a few vertices take a large share of the
// edges (Chung-Lu: 22 % end in 64 of 2^18) the lanes of a warp that meet in one
// word repeat it once each (a PageRank there: 18.8 ms, 9.3 with the replicas).
constexpr int kRankHot = 64;
inline unsigned int rank_smem(unsigned int ns) { return (ns + kRankHot * 32) * 4; }
__device__ __forceinline__ void rank_edges(const AlgoState &st, const RelaxTask &t, const Edge<false> (&ed)[kSteps],
                                           float *acc, unsigned int ns) {
    unsigned int dv[kSteps];
    load_entries<false>(t.src.dst, t.src.dst_bits, ed, dv);
#pragma unroll
    for (int q = 0; q < kSteps; ++q) {
        if (!ed[q].ok) continue;
        const float x = __uint_as_float(ed[q].pay);
        if (dv[q] < kRankHot) atomicAdd(&acc[ns + dv[q] * 32 + (threadIdx.x & 31)], x);
        else if (dv[q] < ns) atomicAdd(&acc[dv[q]], x);
        else atomicAdd(&st.delta[dv[q]], x);
    }
}

template <int BLOCK, bool TB>
__global__ void __launch_bounds__(BLOCK, 1024 / BLOCK) k_relax_rank(AlgoState st, ListArrays la, const Summary *sum,
                                                                    RelaxTask ta, RelaxTask tb, unsigned int ns) {
    extern __shared__ float4 acc4[];
    if (st.loop && !st.loop->work) return;
    float *acc = reinterpret_cast<float *>(acc4);
    unsigned long long kb, ke, zb = 0, eb = 0;
    const RouteView va = task_view(ta, sum, kb, ke);
    RouteView vb{};
    if (TB) vb = task_view(tb, sum, zb, eb);
    if (kb >= ke && zb >= eb) return;
    for (unsigned int i = threadIdx.x; i < (ns + kRankHot * 32) / 4; i += BLOCK) acc4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    LinkCount lc, lb;
    walk_task<kSteps, false, false>(la, va, ta, kb, ke, lc, [&](const Edge<false> (&ed)[kSteps], unsigned long long) {
        rank_edges(st, ta, ed, acc, ns);
    });
    flush_link(lc, ta.link_ctr);
    if (TB) {
        walk_task<kSteps, false, false>(la, vb, tb, zb, eb, lb, [&](const Edge<false> (&ed)[kSteps], unsigned long long) {
            rank_edges(st, tb, ed, acc, ns);
        });
        flush_link(lb, tb.link_ctr);
    }
    __syncthreads();
    for (int v = threadIdx.x >> 5; v < kRankHot; v += BLOCK / 32) {
        float x = acc[ns + v * 32 + (threadIdx.x & 31)];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if ((threadIdx.x & 31) == 0) acc[v] = x;    // ids below kRankHot have no other sum
    }
    __syncthreads();
    float4 *row = reinterpret_cast<float4 *>(st.hub_rep + (size_t)(blockIdx.x % kRankRows) * st.n_hub_rep);
    for (unsigned int i = threadIdx.x; i < ns / 4; i += BLOCK) {
        const float4 x = acc4[i];
        if (x.x != 0.f || x.y != 0.f || x.z != 0.f || x.w != 0.f)
            atomicAdd(i < st.n_hub_rep / 4 ? row + i : reinterpret_cast<float4 *>(st.delta) + i, x);
    }
}

// Two device-sized routes in one launch (cache and zero-copy in the device
// loop, where an iteration's frontier is often a few hundred vertices and a
// launch costs more than the work): the second route's runs follow the
// first's in the warps' order.
template <int ALGO>
__global__ void __launch_bounds__(kRelaxBlock) k_relax_pair(AlgoState st, ListArrays la,
                                                            const Summary *sum, RelaxTask ta,
                                                            RelaxTask tb) {
    if (st.loop && !st.loop->work) return;
    float *hub_rep = st.hub_rep ? st.hub_rep + (size_t)(sm_id() % kHubReplicas) * st.n_hub_rep : nullptr;
    unsigned long long za, zb, ea, eb;
    const RouteView va = task_view(ta, sum, za, ea), vb = task_view(tb, sum, zb, eb);
    const unsigned long long nwarps = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
    const int sh = run_shift(ea + eb, nwarps);
    const unsigned long long na = (ea + (1ull << sh) - 1) >> sh, nb = (eb + (1ull << sh) - 1) >> sh;
    LinkCount la_ct, lb_ct;
    const auto body = [&](const RelaxTask &t) {
        return [&st, &t, hub_rep](const Edge<false> (&ed)[kSteps], unsigned long long) {
            relax_edges<ALGO>(st, t, ed, hub_rep);
        };
    };
    for (unsigned long long r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < na + nb; r += nwarps) {
        if (r < na) walk_run<kSteps, false, ALGO == kSSSP>(la, va, ta, r, sh, 0ull, ea, la_ct, body(ta));
        else walk_run<kSteps, false, ALGO == kSSSP>(la, vb, tb, r - na, sh, 0ull, eb, lb_ct, body(tb));
    }
    flush_link(la_ct, ta.link_ctr);
    flush_link(lb_ct, tb.link_ctr);
}

template <bool WEIGHTS>
__global__ void __launch_bounds__(kRelaxBlock) k_gather(ListArrays la, const Summary *sum,
                                                        RelaxTask t, unsigned int *out_dst,
                                                        unsigned int *out_w, const LoopCtl *loop) {
    if (loop && !loop->work) return;
    unsigned long long kb, ke;
    const RouteView rv = task_view(t, sum, kb, ke);
    LinkCount lc;
    walk_task<kSteps, false, WEIGHTS>(la, rv, t, kb, ke, lc,
                                      [&](const Edge<false> (&ed)[kSteps], unsigned long long k) {
        unsigned int dv[kSteps], wv[kSteps] = {};
        load_entries<false>(t.src.dst, t.src.dst_bits, ed, dv);
        if (WEIGHTS) load_entries<true>(t.src.w, t.src.w_bits, ed, wv);
#pragma unroll
        for (int q = 0; q < kSteps; ++q) {
            if (ed[q].ok) {
                out_dst[k + 32 * q - kb] = dv[q];
                if (WEIGHTS) out_w[k + 32 * q - kb] = wv[q];
            }
        }
    });
    flush_link(lc, t.link_ctr);
}

// Second pass over a resident vertex range (Sec. VI-A: a loaded subgraph is
// processed once more).  Vertices of [vlo, vhi) that became active again
// during this iteration (PageRank: delta > eps; others: frontier bit set and,
// for bucketed SSSP, dist below the bucket) are taken and listed as k_bin
// lists a route's active vertices, and k_relax pushes the list from the
// resident copy: the push touches only the edges of taken vertices, and the
// owner of an edge costs the relax walk's one warp reduction per 32 edges.
// (Before, the push walked every edge of the range and found owners by five
// 64-bit shuffles an edge: 8 M taken of 16.5 M edges, R-MAT 20, took 142 us
// for both launches, now 79 us.)
//
// A block takes 1,024 vertices at a time, a warp 128 of them in four words, so
// that a lane has four residuals, then four offsets, in flight; one atomic
// per block places the entries.
template <int ALGO>
__global__ void __launch_bounds__(kRelaxBlock) k_sp_take(AlgoState st, const unsigned long long *off,
                                                         SecondPassRange r, ListArrays la) {
    if (st.loop) {
        if (!st.loop->work) return;
        st.bucket_limit = st.loop->bucket;
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned int lt_mask = (1u << lane) - 1u;
    unsigned long long done = 0;
    const unsigned long long per_block = 128ull * (kRelaxBlock / 32);
    for (unsigned long long b0 = r.vlo + blockIdx.x * per_block; b0 < r.vhi; b0 += gridDim.x * per_block) {
        const unsigned long long v0 = b0 + 128ull * wid;
        bool take[4];
        float dl[4];
        unsigned int pay[4];
        unsigned long long o0[4], deg[4];
        float hub[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (ALGO == kPR && b0 < st.n_hub_rep) {     // block-uniform
            // the hubs' block sums (k_relax_rank) join their residuals.  What a row
            // gave is taken off it by a reduction, as from delta below, so that
            // other streams' sums stay; all of a lane's loads are in flight
            // together (swapping the rows out waits for each: +7 % of a resident
            // R-MAT 20 PageRank, this +0.3 %).
            float x[4][kRankRows];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const unsigned long long v = v0 + 32 * q + lane;
                const bool in = v < r.vhi && v < st.n_hub_rep;
#pragma unroll
                for (int k = 0; k < kRankRows; ++k)
                    x[q][k] = in ? __ldcg(&st.hub_rep[(size_t)k * st.n_hub_rep + v]) : 0.0f;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int k = 0; k < kRankRows; ++k)
                    if (x[q][k] != 0.0f)
                        atomicAdd(&st.hub_rep[(size_t)k * st.n_hub_rep + (v0 + 32 * q + lane)], -x[q][k]);
#pragma unroll
            for (int w = kRankRows / 2; w > 0; w >>= 1)
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int k = 0; k < w; ++k) x[q][k] += x[q][k + w];
#pragma unroll
            for (int q = 0; q < 4; ++q) hub[q] = x[q][0];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const unsigned long long v = v0 + 32 * q + lane;
            take[q] = false;
            dl[q] = 0.0f;
            pay[q] = 0;
            if (v < r.vhi) {
                if (ALGO == kPR) {
                    if (v < st.n_hub_rep && hub[q] != 0.0f) dl[q] = atomicAdd(&st.delta[v], hub[q]) + hub[q];
                    else dl[q] = __ldcg(&st.delta[v]);
                    take[q] = dl[q] > st.eps;
                } else {
                    take[q] = (__ldcg(&st.bm_cur[v >> 5]) >> (v & 31)) & 1u;
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const unsigned long long v = v0 + 32 * q + lane;
            o0[q] = deg[q] = 0;
            if (take[q]) {
                o0[q] = off[v];
                deg[q] = off[v + 1];
                if (ALGO != kPR) pay[q] = __ldcg(&st.val[v]);
            }
        }
        unsigned int bal[4], cnt[4], n_ent = 0;
        unsigned long long incl[4], eg[4], n_edges = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const unsigned long long v = v0 + 32 * q + lane;
            deg[q] -= o0[q];
            if (take[q]) {
                if (ALGO == kPR) {
                    // Take the delta seen now and subtract it with a reduction,
                    // so that pushes landing on v meanwhile (relaxes of other
                    // streams) stay in delta for later.  No second pass
                    // overlaps this vertex range and k_bin never runs beside
                    // one, so this thread is the only writer of rank[v] now: a
                    // plain update suffices.
                    atomicAdd(&st.delta[v], -dl[q]);
                    rank_add(st, v, st.rank[v], st.rank_lo[v], dl[q]);
                    if (deg[q]) pay[q] = __float_as_uint(st.damping * dl[q] / (float)deg[q]);
                } else if (st.bucket_limit != 0xFFFFFFFFu && pay[q] >= st.bucket_limit) {
                    deg[q] = 0;
                } else {
                    const unsigned int mask = 1u << (v & 31);
                    if (!(atomicAnd(&st.bm_cur[v >> 5], ~mask) & mask)) deg[q] = 0;
                    else pay[q] = __ldcg(&st.val[v]);
                }
            }
            incl[q] = warp_scan_u64(deg[q]);
            bal[q] = __ballot_sync(0xffffffffu, deg[q] > 0);
            cnt[q] = n_ent;
            eg[q] = n_edges;
            n_ent += __popc(bal[q]);
            n_edges += __shfl_sync(0xffffffffu, incl[q], 31);
        }
        unsigned long long block_edges;
        const ListPlace at = block_reserve(n_ent, n_edges, r.cursor, block_edges);
        done += block_edges;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (deg[q] == 0) continue;
            const unsigned long long idx = at.entry + cnt[q] + __popc(bal[q] & lt_mask);
            const unsigned long long eb = at.edge + eg[q] + incl[q] - deg[q];
            const unsigned long long t1 = (eb + deg[q] - 1) / kTile;
            if (idx >= r.vhi - r.vlo || r.tbase + t1 >= la.cap_tiles) {
                atomicOr(la.err, 16u);
                continue;
            }
            la.ebase[r.vlo + idx] = eb;
            la.soff[r.vlo + idx] = o0[q];
            la.pay[r.vlo + idx] = pay[q];
            for (unsigned long long t = (eb + kTile - 1) / kTile; t <= t1; ++t)
                la.tile_first[r.tbase + t] = (unsigned int)idx;
        }
    }
    if (threadIdx.x == 0 && done) atomicAdd(r.edges_out, done);
}

}  // namespace

cudaError_t launch_second_pass(const AlgoState &st, const unsigned long long *off, const SecondPassRange &r,
                               const ListArrays &la, const Summary *sum, cudaStream_t s) {
    if (r.vhi <= r.vlo) return cudaSuccess;
    if ((r.vlo & 31) || r.vhi - r.vlo > kSpEntries || r.E1 - r.E0 > kSpEdgesMax) return cudaErrorInvalidValue;
    const unsigned int tb = sp_take_blocks(r.vhi - r.vlo, 1024);
    switch (st.algo) {
        case kBFS: k_sp_take<kBFS><<<tb, kRelaxBlock, 0, s>>>(st, off, r, la); break;
        case kSSSP: k_sp_take<kSSSP><<<tb, kRelaxBlock, 0, s>>>(st, off, r, la); break;
        case kCC: k_sp_take<kCC><<<tb, kRelaxBlock, 0, s>>>(st, off, r, la); break;
        default: k_sp_take<kPR><<<tb, kRelaxBlock, 0, s>>>(st, off, r, la); break;
    }
    return launch_relax(st, la, sum, sp_push_task(r), r.E1 > r.E0 ? (int)run_blocks(0, r.E1 - r.E0, 8 * device_sms()) : 1, s);
}

// Hub ids that a PageRank relax of at most `edges` edges sums in shared memory,
// a multiple of 4; 0: the plain relax.  Of hub-sorted graphs, with or without
// replicas ("hub_replicas" 0: every sum goes to delta; one addition per edge there
// gave R-MAT 19, resident, an error of 3.8e-6, 152 sums a launch 0.7e-7).  A
// block's sums cost its share of the flush (a vector reduction per 4 ids), so the
// number follows the edges an SM gets.  PageRank, every partition resident, plain
// / 4,096 / 16,384: R-MAT 18 (4.2 M edges) 8.0 / 6.4 / 6.9 ms, R-MAT 19 13.1 / 11.0
// / 9.3, R-MAT 21 37.0 / - / 27.4; R-MAT 12 (65 K edges) 5.4 / 3.2.  The edges of a
// device-sized launch are those of its source, since the host does not know the
// route's: a late iteration with few edges clears and scans the sums all the same.
static unsigned int rank_ids(const AlgoState &st, unsigned long long edges) {
    if ((st.algo != kPR && st.algo != kPPR) || !st.perm || st.V < 4 * kRankHot || edges < kRankNarrow) return 0;
    if (edges >= kRankWide && st.V >= 16384) return 16384;
    return st.V >= 4096 ? 4096u : (unsigned int)st.V & ~3u;
}

// 16,384 ids: one block of 1,024 threads per SM (the cache, and its second
// pass).  Fewer: two blocks of 512, so that another stream's task can have half
// of an SM while this one starts or ends (PPR on R-MAT 24, F tasks of 4 M edges:
// 209 ms, with blocks of 1,024 210 ms, of 256 217 ms).
template <bool TB>
static cudaError_t launch_rank(unsigned int ns, const AlgoState &st, const ListArrays &la, const Summary *sum,
                               const RelaxTask &ta, const RelaxTask &tb, cudaStream_t s) {
    if (ns == 16384) {
        // above the 48 KiB that need no opt-in; the attribute is per device and
        // setting it again is free
        cudaError_t e = cudaFuncSetAttribute(k_relax_rank<1024, TB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)rank_smem(16384));
        if (e != cudaSuccess) return e;
        k_relax_rank<1024, TB><<<device_sms(), 1024, rank_smem(ns), s>>>(st, la, sum, ta, tb, ns);
    } else {
        k_relax_rank<512, TB><<<2 * device_sms(), 512, rank_smem(ns), s>>>(st, la, sum, ta, tb, ns);
    }
    return cudaGetLastError();
}

cudaError_t launch_relax(const AlgoState &st, const ListArrays &la, const Summary *sum,
                         const RelaxTask &t, int grid_cap, cudaStream_t s) {
    // edges that the task can have at most: its host bounds, or its source's
    const unsigned long long most =
        !t.device_sized && !t.dev_edge ? (t.k_end > t.k_begin ? t.k_end - t.k_begin : 0ull)
        : t.route == kRouteZ && !t.sp_cursor ? 0ull : t.src.e_hi - t.src.e_lo;
    if (const unsigned int ns = rank_ids(st, most)) return launch_rank<false>(ns, st, la, sum, t, t, s);
    unsigned int grid = (unsigned int)grid_cap;
    if (!t.device_sized && !t.dev_edge) {
        if (t.k_begin >= t.k_end) return t.sp_reset ? cudaMemsetAsync(t.sp_reset, 0, 8, s) : cudaSuccess;
        grid = run_blocks(t.k_begin, t.k_end, grid);
    }
    switch (st.algo) {
        case kBFS: k_relax<kBFS><<<grid, kRelaxBlock, 0, s>>>(st, la, sum, t); break;
        case kSSSP: k_relax<kSSSP><<<grid, kRelaxBlock, 0, s>>>(st, la, sum, t); break;
        case kCC: k_relax<kCC><<<grid, kRelaxBlock, 0, s>>>(st, la, sum, t); break;
        default: k_relax<kPR><<<grid, kRelaxBlock, 0, s>>>(st, la, sum, t); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_relax_pair(const AlgoState &st, const ListArrays &la, const Summary *sum,
                              const RelaxTask &ta, const RelaxTask &tb, int grid, cudaStream_t s) {
    if (const unsigned int ns = rank_ids(st, ta.src.e_hi - ta.src.e_lo)) return launch_rank<true>(ns, st, la, sum, ta, tb, s);
    switch (st.algo) {
        case kBFS: k_relax_pair<kBFS><<<grid, kRelaxBlock, 0, s>>>(st, la, sum, ta, tb); break;
        case kSSSP: k_relax_pair<kSSSP><<<grid, kRelaxBlock, 0, s>>>(st, la, sum, ta, tb); break;
        case kCC: k_relax_pair<kCC><<<grid, kRelaxBlock, 0, s>>>(st, la, sum, ta, tb); break;
        default: k_relax_pair<kPR><<<grid, kRelaxBlock, 0, s>>>(st, la, sum, ta, tb); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_gather(const ListArrays &la, const Summary *sum, const RelaxTask &t,
                          unsigned int *out_dst, unsigned int *out_w, int grid_cap,
                          cudaStream_t s, const LoopCtl *loop) {
    unsigned int grid = (unsigned int)grid_cap;
    if (!t.device_sized && !t.dev_edge) {
        if (t.k_begin >= t.k_end) return cudaSuccess;
        grid = run_blocks(t.k_begin, t.k_end, grid);
    }
    if (out_w) k_gather<true><<<grid, kRelaxBlock, 0, s>>>(la, sum, t, out_dst, out_w, loop);
    else k_gather<false><<<grid, kRelaxBlock, 0, s>>>(la, sum, t, out_dst, out_w, loop);
    return cudaGetLastError();
}

}  // namespace hytg
