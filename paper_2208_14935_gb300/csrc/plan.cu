// Cost-aware task generation on the device (Sec. V-A, Alg. 1, cost part):
//   k_count   frontier bitmap -> per-partition |A_i|, active edges and
//             128-byte lines (footnote to Eq. 3);
//   k_select  one block: the engine of every partition from Eq. 1-3 and the
//             selection rule, then the prefix sums that give each partition
//             its place in its route's list (Alg. 1 gathers the C and the Z
//             partitions into one batch each on the GPU);
//   k_bin     writes the route lists (edge base, row offset, pushed value)
//             and the tile index of the load-balanced relax kernels, takes the
//             delta of delta-PageRank, and clears the bits it consumed.
// A partition's slice of its route list is filled through one 64-bit cursor
// per partition (entries in the low 24 bits, edges above), so a warp
// reserves the entry range and the edge range of its 128 vertices in one
// atomic.  In the device loop k_select also takes the loop's decision.
//
// Bucketed SSSP (delta-stepping): with a bucket limit B, only active
// vertices with dist < B are eligible; the others stay set in the bitmap and
// are counted as pending, with their smallest distance, for the next bucket.
#include "common.cuh"
#include "cost_model.cuh"
#include "hytg.h"

namespace hytg {

namespace {

// The bitmap walk.  A unit is 4 consecutive words (one 16-byte load, 128
// vertices); a chunk is `cw` words (a power of two from 4 to 128), which one
// warp loads with cw / 4 lanes.  A warp takes chunks warp, warp + nwarps, ...,
// kPrefetch of them at a time so that their latencies overlap, and then
// visits the units that hold any bit; a sparse frontier skips the rest.
// body(w0, x) sees the unit's first word index and its words, the same in
// every lane (reloaded: a cache hit).  The walk only reads the bitmap; body
// may rewrite its own unit's words.  The bitmap is padded to a multiple of
// 32 words, so a unit is wholly inside it.
//
// The chunk size is the launcher's (walk_chunk): a dense unit costs a few
// microseconds of dependent loads, atomics and stores, so what bounds the
// walk is how many units one warp visits in turn.  With whole 128-word chunks
// a graph of 2^20 vertices (R-MAT 20, half of them active) kept 256 warps
// busy with 32 units each; chunks of 4 words spread them over every warp:
// k_bin 140 -> 20 us, k_count 93 -> about 15 us.  At 2^24 vertices (R-MAT 24,
// 44 % active) k_bin went from 313 to 129 us, k_count from 206 to about 50 us.
constexpr int kPrefetch = 8;
template <class F>
__device__ __forceinline__ void for_units(const unsigned int *bm, unsigned int n_words, unsigned int cw,
                                          F &&body) {
    const unsigned int lane = threadIdx.x & 31;
    const unsigned int nwarps = gridDim.x * (blockDim.x >> 5);
    const unsigned int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const unsigned int lanes = cw / 4, n_units = n_words / 4;
    const unsigned int n_chunks = (n_words + cw - 1) / cw;
    const uint4 *bm4 = reinterpret_cast<const uint4 *>(bm);
    for (unsigned int c0 = w; c0 < n_chunks; c0 += nwarps * kPrefetch) {
        uint4 pre[kPrefetch];
#pragma unroll
        for (int j = 0; j < kPrefetch; ++j) {
            const unsigned int c = c0 + j * nwarps, u = c * lanes + lane;
            pre[j] = (lane < lanes && c < n_chunks && u < n_units) ? bm4[u] : make_uint4(0u, 0u, 0u, 0u);
        }
        unsigned int mine = 0;                      // lane j: the live units of chunk c0 + j * nwarps
#pragma unroll
        for (int j = 0; j < kPrefetch; ++j) {
            const unsigned int nz = __ballot_sync(0xffffffffu, (pre[j].x | pre[j].y | pre[j].z | pre[j].w) != 0u);
            if (lane == (unsigned int)j) mine = nz;
        }
        unsigned int live = __ballot_sync(0xffffffffu, mine != 0u);
        while (live) {                              // warp-uniform
            const int j = __ffs(live) - 1;
            live &= live - 1;
            unsigned int m = __shfl_sync(0xffffffffu, mine, j);
            while (m) {
                const unsigned int u = (c0 + j * nwarps) * lanes + (__ffs(m) - 1);
                m &= m - 1;
                body(u * 4, bm4[u]);
            }
        }
    }
}

// Partition holding bitmap word `widx` (bounds are word indices): the
// partition of the word's 32-word round from the round table, then forward
// over the partition bounds inside the round (partitions are whole words, so
// at most 31 steps, in practice none or one).
__device__ __forceinline__ unsigned int find_part(const GraphDev &g, unsigned int widx) {
    unsigned int p = __ldg(&g.round_part[widx >> 5]);
    while (p + 1 < g.N && __ldg(&g.part_wb[p + 1]) <= widx) ++p;
    return p;
}

// Counts of one partition gathered by a warp; edges, lines and prio are
// per-lane sums, reduced only when they are flushed.
struct CountAcc {
    unsigned int nact = 0, ent = 0;
    unsigned long long edges = 0, lines = 0, prio = 0;
};
__device__ __forceinline__ void flush_count(const PartArrays &pa, unsigned int p, CountAcc &a, bool prio) {
    if (p != 0xFFFFFFFFu && a.nact) {               // warp-uniform
        const unsigned int ent = __reduce_add_sync(0xffffffffu, a.ent);
        const unsigned long long edges = warp_sum_u64(a.edges), lines = warp_sum_u64(a.lines);
        const unsigned long long pr = prio ? warp_sum_u64(a.prio) : 0ull;
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&pa.n_act[p], (unsigned long long)a.nact);
            if (ent) {
                atomicAdd(&pa.entries[p], (unsigned long long)ent);
                atomicAdd(&pa.edges[p], edges);
                atomicAdd(&pa.lines[p], lines);
            }
            if (pr) atomicAdd(&pa.prio[p], pr);
        }
    }
    a = CountAcc();
}

// m_shift: log2 of the request size m when it is a power of two (a 64-bit
// division per vertex otherwise), else -1.
__global__ void __launch_bounds__(256) k_count(GraphDev g, AlgoState st, PartArrays pa,
                                               unsigned long long m, int m_shift, unsigned int cw) {
    if (st.loop) st.bucket_limit = st.loop->bucket;
    const int lane = threadIdx.x & 31;
    const bool bucketed = st.bucket_limit != 0xFFFFFFFFu;
    unsigned long long pend = 0;
    unsigned int pend_min = 0xFFFFFFFFu;
    unsigned int cur_p = 0xFFFFFFFFu, p_lo = 1, p_hi = 0;   // word range of cur_p
    CountAcc acc;
    for_units(st.bm_cur, (unsigned int)g.n_words_alloc, cw, [&](unsigned int w0, uint4 x) {
        const unsigned int wq[4] = {x.x, x.y, x.z, x.w};
        unsigned long long o0[4], o1[4];
        unsigned int dv[4];
        float dl[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            o0[q] = o1[q] = 0;
            dv[q] = 0;
            dl[q] = 0.f;
            if ((wq[q] >> lane) & 1u) {
                const unsigned long long v = (unsigned long long)(w0 + q) * 32 + lane;
                o0[q] = g.off[v];
                o1[q] = g.off[v + 1];
                if (bucketed) dv[q] = st.val[v];
                if (st.prio) dl[q] = st.delta[v];
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (wq[q] == 0) continue;              // warp-uniform
            const unsigned int widx = w0 + q;
            bool act = (wq[q] >> lane) & 1u;
            unsigned int elig = wq[q];
            if (bucketed) {
                if (act && dv[q] >= st.bucket_limit) {
                    ++pend;
                    pend_min = min(pend_min, dv[q]);
                    act = false;
                }
                elig = __ballot_sync(0xffffffffu, act);
                if (elig == 0) continue;
            }
            if (widx < p_lo || widx >= p_hi) {
                flush_count(pa, cur_p, acc, st.prio);
                cur_p = find_part(g, widx);
                p_lo = g.part_wb[cur_p];
                p_hi = g.part_wb[cur_p + 1];
            }
            acc.nact += __popc(elig);
            if (act && o1[q] > o0[q]) {
                const unsigned long long deg = o1[q] - o0[q];
                acc.ent += 1;
                acc.edges += deg;
                const unsigned long long ln =
                    m_shift >= 0 ? ((o1[q] * 4ull - 1) >> m_shift) - ((o0[q] * 4ull) >> m_shift) + 1
                                 : lines_spanned(o0[q] * 4ull, deg * 4ull, m);
                acc.lines += st.n_arrays * ln;
            }
            if (st.prio && act) {
                // |delta| in units of 2^-24, capped at 2^40 per vertex; the
                // sum only orders the F tasks, so rounding cannot matter
                acc.prio += (unsigned long long)fminf(fabsf(dl[q]) * 16777216.f, 1099511627776.f);
            }
        }
    });
    flush_count(pa, cur_p, acc, st.prio);
    if (bucketed) {
        pend = warp_sum_u64(pend);
        pend_min = __reduce_min_sync(0xffffffffu, pend_min);
        if (lane == 0 && pend) {
            atomicAdd(pa.pending, pend);
            atomicMax(pa.pending_inv, (unsigned long long)(~pend_min));   // max of ~d = ~min d
        }
    }
}

// ------------------------------------------------------------- k_select
// One block: routes, per-route prefixes over partitions, the summary and, in
// the device loop, the loop's decision.  What bounds it is latency (loads,
// the cost model's divisions, the scan, a handful of stores), so the block is
// as small as the partitions allow (one warp for up to 32), the cost model
// divides in 64 bits, and the loop's decision runs here instead of in a
// kernel of its own (a launch of about 5 us per device iteration; k_select
// itself took 10 us).
constexpr int kSelScan = 8;           // entries and edges of routes 1..4: prefixes
constexpr int kSelVals = 17;          // + lines (4), partitions (4) of routes 1..4, active vertices

__device__ void loop_decide(const Summary *sum, LoopCtl *ctl, unsigned long long cond);

__global__ void __launch_bounds__(kSelectBlock) k_select(GraphDev g, PartArrays pa, CostParams cp,
                                                         Summary *sum, LoopCtl *ctl,
                                                         unsigned long long cond) {
    __shared__ unsigned long long s_w[kSelectBlock / 32][kSelVals];
    __shared__ unsigned long long s_tot[kSelVals];
    const unsigned int N = g.N;
    const unsigned int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
    // per-route sums over this thread's contiguous chunk of partitions
    const unsigned int ppt = (N + nt - 1) / nt;
    const unsigned int p0 = min(N, tid * ppt), p1 = min(N, p0 + ppt);
    unsigned long long v[kSelVals];
#pragma unroll
    for (int q = 0; q < kSelVals; ++q) v[q] = 0;
    for (unsigned int p = p0; p < p1; ++p) {
        const unsigned long long act = pa.n_act[p], ent = pa.entries[p], edg = pa.edges[p], lin = pa.lines[p];
        const int r = decide_route_counts(p, g.part_eb[p + 1] - g.part_eb[p], act, edg, lin, cp);
        pa.route[p] = (unsigned char)r;
        // compile-time indices keep v[] in registers; a partition without a
        // route has no entries, edges or lines
#pragma unroll
        for (int q = 1; q < kRoutes; ++q) {
            if (r == q) {
                v[q - 1] += ent;
                v[3 + q] += edg;
                v[7 + q] += lin;
                v[11 + q] += 1;
            }
        }
        v[16] += act;
    }
    unsigned long long ex[kSelScan];                // exclusive prefixes of this thread
#pragma unroll
    for (int q = 0; q < kSelScan; ++q) {
        const unsigned long long incl = warp_scan_u64(v[q]);
        ex[q] = incl - v[q];
        if (lane == 31) s_w[wid][q] = incl;
    }
#pragma unroll
    for (int q = kSelScan; q < kSelVals; ++q) {
        const unsigned long long t = warp_sum_u64(v[q]);
        if (lane == 0) s_w[wid][q] = t;
    }
    __syncthreads();
    if (tid < kSelVals) {
        unsigned long long run = 0;
        for (unsigned int w = 0; w < nw; ++w) {
            const unsigned long long t = s_w[w][tid];
            s_w[w][tid] = run;
            run += t;
        }
        s_tot[tid] = run;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kSelScan; ++q) ex[q] += s_w[wid][q];
    for (unsigned int p = p0; p < p1; ++p) {
        const int r = pa.route[p];
        const unsigned long long ent = pa.entries[p], edg = pa.edges[p];
        unsigned long long re = 0, rg = 0;
#pragma unroll
        for (int q = 1; q < kRoutes; ++q) {
            if (r == q) {
                re = ex[q - 1];
                rg = ex[3 + q];
                ex[q - 1] += ent;
                ex[3 + q] += edg;
            }
        }
        pa.route_entry[p] = re;
        pa.route_edge[p] = rg;
    }
    __shared__ Summary s_sum;                       // the summary, also read by the decision
    if (tid < kRoutes) {
        // thread r writes route r's totals and bases
        const unsigned int r = tid;
        unsigned long long e = 0, t = 0, parts = 0;
        for (unsigned int q = 1; q < kRoutes; ++q) {
            if (q < r) {
                e += s_tot[q - 1];
                t += (s_tot[3 + q] + kTile - 1) / kTile;
            }
            parts += s_tot[11 + q];
        }
        s_sum.route_entries[r] = r ? s_tot[r - 1] : 0ull;
        s_sum.route_edges[r] = r ? s_tot[3 + r] : 0ull;
        s_sum.route_lines[r] = r ? s_tot[7 + r] : 0ull;
        s_sum.route_parts[r] = (unsigned int)(r ? s_tot[11 + r] : N - parts);
        s_sum.route_entry_base[r] = e;
        s_sum.route_tile_base[r] = t;
    }
    if (tid == kRoutes) {
        s_sum.n_active = s_tot[16];
        s_sum.pending = *pa.pending;
        s_sum.pending_min = ~(unsigned int)(*pa.pending_inv);
        s_sum.alive = pa.alive ? *pa.alive : 0ull;
    }
    __syncthreads();
    for (unsigned int i = tid; i < sizeof(Summary) / 4; i += nt)
        reinterpret_cast<unsigned int *>(sum)[i] = reinterpret_cast<const unsigned int *>(&s_sum)[i];
    if (ctl) loop_decide(&s_sum, ctl, cond);
}

// ------------------------------------------------------ device loop
// Thread 0: the host loop's decisions for the iteration just planned.
__device__ void loop_decide_one(const Summary *sum, LoopCtl *ctl, cudaGraphConditionalHandle h) {
    ctl->work = 0;
    ctl->tail = 0;
    ++ctl->bodies;
    if (sum->n_active == 0) {
        if (sum->pending == 0) {
            ctl->status = kLoopDone;
            cudaGraphSetConditional(h, 0);
            return;
        }
        // the current bucket is settled: open the next one at the smallest
        // pending distance (delta-stepping), and plan again
        unsigned long long nb = (unsigned long long)(ctl->bucket > sum->pending_min ? ctl->bucket : sum->pending_min);
        nb += ctl->delta;
        ctl->bucket = nb < 0xFFFFFFFEull ? (unsigned int)nb : 0xFFFFFFFEu;
        if (sum->pending_min >= 0xFFFFFFFEu) ctl->bucket = 0xFFFFFFFFu;
        ++ctl->it;
        cudaGraphSetConditional(h, 1);
        return;
    }
    if ((unsigned long long)ctl->it >= ctl->max_it) {
        ctl->status = kLoopMaxIt;
        cudaGraphSetConditional(h, 0);
        return;
    }
    if (ctl->cancel && *ctl->cancel != 0u) {
        ctl->status = kLoopCancel;        // nothing of this iteration runs
        cudaGraphSetConditional(h, 0);
        return;
    }
    unsigned long long act = 0;
    for (int q = 0; q < kRoutes; ++q) act += sum->route_edges[q];
    if (ctl->tail_ok && ctl->it >= ctl->tail_not && ctl->n_rec < ctl->rec_cap && sum->n_active <= kTailActive &&
        act <= kTailEdges && sum->n_active + sum->pending <= kTailQueue && sum->route_parts[kRouteF] == 0 &&
        (sum->route_parts[kRouteC] == 0 || ctl->tail_gather)) {
        ctl->tail = 1;                    // k_tail runs it, and those that follow
        cudaGraphSetConditional(h, 1);
        return;
    }
    const bool f_host = sum->route_parts[kRouteF] != 0 && !ctl->f_handles;
    const bool c_host = sum->route_parts[kRouteC] != 0 &&
                        (!ctl->c_handle || sum->route_edges[kRouteC] > ctl->c_cap);
    if (f_host || c_host || ctl->n_rec >= ctl->rec_cap) {
        ctl->status = kLoopHost;          // the host takes this iteration from k_bin on
        cudaGraphSetConditional(h, 0);
        return;
    }
    hytg_iter_record *r = (hytg_iter_record *)ctl->rec + ctl->n_rec++;
    for (int q = 0; q < kRoutes; ++q) {
        r->route_partitions[q] = sum->route_parts[q];
        r->route_edges[q] = sum->route_edges[q];
        ctl->route_parts[q] += sum->route_parts[q];
        ctl->route_entries[q] += sum->route_entries[q];
        ctl->route_edges[q] += sum->route_edges[q];
    }
    r->active_vertices = sum->n_active;
    r->active_edges = act;
    r->f_tasks = 0;
    r->link_bytes = sum->route_lines[kRouteZ] * ctl->m;
    r->device_ms = 0.0;
    ctl->z_lines += sum->route_lines[kRouteZ];
    ctl->vertices += sum->n_active;
    ctl->edges += act;
    ++ctl->iterations;
    ctl->work = 1;
    ++ctl->it;
    cudaGraphSetConditional(h, 1);
}

// The whole block: the decision, then the IF nodes of the partitions routed F
// (each copies its partition into a staging slot and relaxes it) and of the
// C route.
__device__ void loop_decide(const Summary *sum, LoopCtl *ctl, unsigned long long cond) {
    __shared__ unsigned long long s_parts, s_bytes;
    if (threadIdx.x == 0) {
        s_parts = s_bytes = 0;
        loop_decide_one(sum, ctl, (cudaGraphConditionalHandle)cond);
    }
    __syncthreads();
    // every IF condition is set on every iteration (a value set once would
    // otherwise carry over to the next iteration of the loop), and left
    // closed when the device does not take the iteration
    const bool work = ctl->work != 0;
    if (ctl->f_handles) {
        unsigned long long np = 0, nb = 0;
        for (unsigned int i = threadIdx.x; i < ctl->n_parts; i += blockDim.x) {
            const bool f = work && ctl->route[i] == kRouteF;
            cudaGraphSetConditional((cudaGraphConditionalHandle)ctl->f_handles[i], f ? 1u : 0u);
            if (f) {
                ++np;
                const unsigned long long e0 = ctl->part_eb[i], n = ctl->part_eb[i + 1] - e0;
                nb += 4 * word_span(e0, n, ctl->dst_bits).n;
                if (ctl->w_bits) nb += 4 * word_span(e0, n, ctl->w_bits).n;
            }
        }
        if (np) {
            atomicAdd(&s_parts, np);
            atomicAdd(&s_bytes, nb);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const bool c_on = work && sum->route_edges[kRouteC] != 0;
        if (ctl->c_handle) cudaGraphSetConditional((cudaGraphConditionalHandle)ctl->c_handle, c_on ? 1u : 0u);
        if (work) {
            hytg_iter_record *r = (hytg_iter_record *)ctl->rec + (ctl->n_rec - 1);
            r->f_tasks = (unsigned int)s_parts;
            r->link_bytes += s_bytes;
            ctl->f_parts += s_parts;
            ctl->f_bytes += s_bytes;
            if (c_on && ctl->c_handle) {
                ++ctl->c_iters;
                ctl->c_lines += sum->route_lines[kRouteC];
                r->link_bytes += sum->route_lines[kRouteC] * ctl->m;
            }
        }
    }
}

// ---------------------------------------------------------------- k_bin
// MODE: what an entry carries.  A unit's entries and edges are placed with
// one atomic on its partition's cursor (one per partition if the unit spans a
// bound), issued once the unit's four words are scanned, so its latency is
// paid per 128 vertices instead of per 32.
enum BinMode : int { kBinVal = 0, kBinPR = 1, kBinBatch = 2 };

template <int MODE>
__global__ void __launch_bounds__(256) k_bin(GraphDev g, AlgoState st, PartArrays pa, ListArrays la,
                                             const Summary *sum, unsigned int cw) {
    if (st.loop) {
        if (!st.loop->work) return;
        st.bucket_limit = st.loop->bucket;
    }
    const int lane = threadIdx.x & 31;
    const unsigned int lt_mask = (1u << lane) - 1u;
    const bool bucketed = MODE == kBinVal && st.bucket_limit != 0xFFFFFFFFu;
    unsigned long long work = 0;
    unsigned int cur_p = 0xFFFFFFFFu, p_lo = 1, p_hi = 0;
    unsigned long long rbase = 0, tbase = 0, pe0 = 0, pg0 = 0;
    for_units(st.bm_cur, (unsigned int)g.n_words_alloc, cw, [&](unsigned int w0, uint4 x) {
        const unsigned int wq[4] = {x.x, x.y, x.z, x.w};
        unsigned int elig[4];
        unsigned long long o0[4], deg[4];
        unsigned int vv[4];
        float rk[4], rl[4];
        unsigned long long bf[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            o0[q] = deg[q] = 0;
            vv[q] = 0;
            rk[q] = rl[q] = 0.0f;
            bf[q] = 0;
            if ((wq[q] >> lane) & 1u) {
                const unsigned long long v = (unsigned long long)(w0 + q) * 32 + lane;
                o0[q] = g.off[v];
                deg[q] = g.off[v + 1];
                if (MODE == kBinBatch) bf[q] = st.batch_mode == kBatchPPR ? st.b_fr32[v] : st.b_fr[v];
                else if (MODE == kBinPR) {
                    vv[q] = __float_as_uint(st.delta[v]);
                    rk[q] = st.rank[v];
                    rl[q] = st.rank_lo[v];
                }
                else vv[q] = st.val[v];
            }
        }
        unsigned int any = 0;                      // bit q: word q has an eligible vertex
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            elig[q] = bucketed ? __ballot_sync(0xffffffffu, ((wq[q] >> lane) & 1u) && vv[q] < st.bucket_limit)
                               : wq[q];
            if (elig[q]) any |= 1u << q;
            deg[q] = ((elig[q] >> lane) & 1u) ? deg[q] - o0[q] : 0ull;
        }
        // the unit's eligible bits are consumed; the rest wait for a later bucket
        if (lane == 0 && any)
            reinterpret_cast<uint4 *>(st.bm_cur)[w0 / 4] = make_uint4(wq[0] & ~elig[0], wq[1] & ~elig[1],
                                                                      wq[2] & ~elig[2], wq[3] & ~elig[3]);
        unsigned long long incl[4];
        unsigned int bal[4];
        if (__all_sync(0xffffffffu, (deg[0] | deg[1] | deg[2] | deg[3]) < (1ull << 27))) {
            unsigned int y[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) y[q] = (unsigned int)deg[q];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const unsigned int t = __shfl_up_sync(0xffffffffu, y[q], o);
                    if (lane >= o) y[q] += t;
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) incl[q] = y[q];
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) incl[q] = warp_scan_u64(deg[q]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) bal[q] = __ballot_sync(0xffffffffu, deg[q] > 0);
        while (any) {                              // once per partition of the unit
            const unsigned int wf = w0 + (__ffs(any) - 1);
            if (wf < p_lo || wf >= p_hi) {
                cur_p = find_part(g, wf);
                p_lo = g.part_wb[cur_p];
                p_hi = g.part_wb[cur_p + 1];
                const int rp = pa.route[cur_p];
                rbase = sum->route_entry_base[rp];
                tbase = sum->route_tile_base[rp];
                pe0 = pa.route_entry[cur_p];
                pg0 = pa.route_edge[cur_p];
            }
            unsigned int cnt[4];                   // entries and edges before word q
            unsigned long long eg[4], n_edges = 0;
            unsigned int n_ent = 0, here = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const bool in = ((any >> q) & 1u) && w0 + q < p_hi;
                cnt[q] = n_ent;
                eg[q] = n_edges;
                if (in) {
                    here |= 1u << q;
                    n_ent += __popc(bal[q]);
                    n_edges += __shfl_sync(0xffffffffu, incl[q], 31);
                }
            }
            any &= ~here;
            unsigned long long old = 0;
            if (lane == 0 && n_ent) old = atomicAdd(&pa.cursor[cur_p], (n_edges << 24) | (unsigned long long)n_ent);
            if (MODE == kBinPR) {
                // take the accumulated delta (Sec. VI-A delta-based PageRank)
                // while the cursor's value is on its way
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (((here >> q) & 1u) && ((elig[q] >> lane) & 1u)) {
                        const unsigned long long v = (unsigned long long)(w0 + q) * 32 + lane;
                        const float dl = __uint_as_float(vv[q]);
                        st.delta[v] = 0.0f;
                        rank_add(st, v, rk[q], rl[q], dl);
                        vv[q] = __float_as_uint(deg[q] ? st.damping * dl / (float)deg[q] : 0.0f);
                    }
                }
            }
            old = __shfl_sync(0xffffffffu, old, 0);
            const unsigned long long ent0 = rbase + pe0 + (old & 0xFFFFFFull), edge0 = pg0 + (old >> 24);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (!((here >> q) & 1u) || deg[q] == 0) continue;
                const unsigned long long idx = ent0 + cnt[q] + __popc(bal[q] & lt_mask);
                const unsigned long long eb = edge0 + eg[q] + (incl[q] - deg[q]);
                const unsigned long long t0 = (eb + kTile - 1) / kTile;
                const unsigned long long t1 = (eb + deg[q] - 1) / kTile;
                if (idx >= la.cap_entries || (t0 <= t1 && tbase + t1 >= la.cap_tiles)) {
                    atomicOr(la.err, 2u);
                } else {
                    la.ebase[idx] = eb;
                    la.soff[idx] = o0[q];
                    la.pay[idx] = MODE == kBinBatch ? 0u : vv[q];
                    if (MODE == kBinBatch) {
                        la.pay64[idx] = bf[q];
                        la.vid[idx] = (unsigned int)((w0 + q) * 32 + lane);
                        work += (unsigned long long)__popcll(bf[q]) * deg[q];
                    }
                    const unsigned int rel = (unsigned int)(idx - rbase);
                    for (unsigned long long t = t0; t <= t1; ++t) la.tile_first[tbase + t] = rel;
                }
            }
        }
    });
    if (MODE == kBinBatch) {
        work = warp_sum_u64(work);
        if (lane == 0 && work) atomicAdd(st.src_work, work);
    }
}

}  // namespace

// Blocks of 256 threads that fit on the device at once for `kernel`.
template <class K>
unsigned long long resident_blocks(K kernel) {
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 256, 0) != cudaSuccess ||
        sms <= 0 || per_sm <= 0)
        return 2ull * device_sms();
    return (unsigned long long)sms * (unsigned long long)per_sm;
}

// Chunk size and grid of a bitmap walk (see for_units): the largest chunk, up
// to 128 words, that still gives every resident warp four, so that warps end
// within a quarter of one another, but at least 4 words; then one resident
// wave, at most one chunk per warp.
struct WalkGrid {
    unsigned int cw, blocks;
};
WalkGrid walk_grid(unsigned long long n_words, unsigned long long resident) {
    unsigned int cw = 128;
    while (cw > 4 && n_words / cw < 4 * 8 * resident) cw >>= 1;
    const unsigned long long blocks = ((n_words + cw - 1) / cw + 7) / 8;
    return {cw, (unsigned int)(blocks < resident ? blocks : resident)};
}

cudaError_t launch_count(const GraphDev &g, const AlgoState &st, const PartArrays &pa,
                         unsigned long long m, cudaStream_t s) {
    if (g.n_words_alloc == 0) return cudaSuccess;
    static const unsigned long long resident = resident_blocks(k_count);
    const WalkGrid w = walk_grid(g.n_words_alloc, resident);
    k_count<<<w.blocks, 256, 0, s>>>(g, st, pa, m, log2_exact(m), w.cw);
    return cudaGetLastError();
}

cudaError_t launch_select(const GraphDev &g, const PartArrays &pa, const CostParams &cp,
                          Summary *sum, cudaStream_t s, LoopCtl *ctl, unsigned long long cond) {
    unsigned int threads = (g.N + 31) / 32 * 32;
    if (threads > (unsigned int)kSelectBlock) threads = kSelectBlock;
    if (threads < 32) threads = 32;
    k_select<<<1, threads, 0, s>>>(g, pa, cp, sum, ctl, cond);
    return cudaGetLastError();
}

cudaError_t launch_bin(const GraphDev &g, const AlgoState &st, const PartArrays &pa,
                       const ListArrays &la, const Summary *sum, cudaStream_t s) {
    if (g.n_words_alloc == 0) return cudaSuccess;
    static const unsigned long long res_val = resident_blocks(k_bin<kBinVal>);
    static const unsigned long long res_pr = resident_blocks(k_bin<kBinPR>);
    static const unsigned long long res_batch = resident_blocks(k_bin<kBinBatch>);
    if (st.batch_mode != kBatchNone) {
        const WalkGrid w = walk_grid(g.n_words_alloc, res_batch);
        k_bin<kBinBatch><<<w.blocks, 256, 0, s>>>(g, st, pa, la, sum, w.cw);
    } else if (st.algo == kPR || st.algo == kPPR) {
        const WalkGrid w = walk_grid(g.n_words_alloc, res_pr);
        k_bin<kBinPR><<<w.blocks, 256, 0, s>>>(g, st, pa, la, sum, w.cw);
    } else {
        const WalkGrid w = walk_grid(g.n_words_alloc, res_val);
        k_bin<kBinVal><<<w.blocks, 256, 0, s>>>(g, st, pa, la, sum, w.cw);
    }
    return cudaGetLastError();
}

}  // namespace hytg
