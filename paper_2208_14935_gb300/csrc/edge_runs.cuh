// The load-balanced walk over a route's active edges, shared by the relax,
// gather and batched relax kernels.
//
// The active vertices of a route form a list; their out-edges, in list order,
// form the route's edge space.  A warp takes a run of up to kRun consecutive
// route edges.  The tile index written by k_bin gives the entry that owns the first
// edge of the run's tile (kTile edges); the run's own first entry is found by
// probing the tile's entries 32 at a time.  The warp then loads a window of 32
// entries, one per lane (first edge, row offset, pushed value), and steps over
// the window's edges 32 at a time: the lanes whose list starts inside the step
// set one bit each (redux.or), and a lane's owner is the number of lists that
// start at or before its edge (a popcount), so three or four shuffles give
// every edge its address and value.  No shared memory and no block barrier:
// what bounds the relax kernels, away from the reduction rate of the L2, is
// the latency of list -> edge -> value -> reduction, which independent warps
// overlap.  A run is 256 edges, or fewer when a task has fewer runs than the
// launch has warps; an index entry per run instead of per tile made k_bin
// two to four times slower (20 -> 42 us on R-MAT 20, half of it active).
// Against blocks that set up tiles of 2,048 edges in shared memory, with four
// barriers a tile: a PageRank relax of 16.5 M resident edges takes the same
// 115 us (143 G reductions/s, the L2's rate), BFS on a 1021 x 1031 mesh
// (frontiers of a few hundred vertices) went from 41.6 to 32.7 ms, serving 24
// SSSP queries on 4 M edges from 8.4 to 7.3 ms.
#pragma once

#include "common.cuh"

namespace hytg {

__device__ __forceinline__ unsigned int sm_id() {
    unsigned int id;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(id));
    return id;
}

// Where a task's list lies: the route's first entry and tile, its entries and
// edges.
struct RouteView {
    unsigned long long rbase, tbase, n_ent, n_edges;
};

// The task's edge range [kb, ke) in its route's edge space: the host's bounds,
// the whole route (device_sized), or one partition's slice of the F route
// read on the device (dev_edge; its first list entry goes to t.first_entry),
// or a second pass's list.
__device__ __forceinline__ RouteView task_view(RelaxTask &t, const Summary *sum, unsigned long long &kb,
                                               unsigned long long &ke) {
    RouteView rv;
    if (t.sp_cursor) {
        const unsigned long long c = *t.sp_cursor;
        rv = {t.sp_rbase, t.sp_tbase, c & kSpEntries, c >> 30};
        kb = 0;
        ke = rv.n_edges;
        return rv;
    }
    if (t.sp_reset && blockIdx.x == 0 && threadIdx.x == 0) *t.sp_reset = 0ull;
    rv.rbase = sum->route_entry_base[t.route];
    rv.tbase = sum->route_tile_base[t.route];
    rv.n_ent = sum->route_entries[t.route];
    rv.n_edges = sum->route_edges[t.route];
    if (t.dev_edge) {
        kb = *t.dev_edge;
        ke = kb + *t.dev_len;
        t.first_entry = *t.dev_entry;
    } else if (t.device_sized) {
        kb = 0;
        ke = sum->route_edges[t.route];
    } else {
        kb = t.k_begin;
        ke = t.k_end;
    }
    return rv;
}

// Host-link reads of a task that reads mapped host memory: the 32-byte sectors
// and 128-byte lines that its edges' entries occupy in each array read (base
// 256-byte aligned).  The edges of an entry are at increasing addresses, so a
// sector (line) is new where it differs from the one the previous edge ended
// in; a run's first edge is compared with the edge before it.  Per-lane
// counts, added once per warp.
struct LinkCount {
    unsigned int sec = 0, ln = 0;
};
__device__ __forceinline__ void count_link(LinkCount &lc, long long e, long long prev, unsigned int bits) {
    const unsigned long long a = (unsigned long long)e * bits, z = a + bits - 1;
    const unsigned long long p = prev < 0 ? ~0ull : (unsigned long long)prev * bits + bits - 1;
    lc.sec += ((a >> 8) != (p >> 8)) + ((z >> 8) != (a >> 8));
    lc.ln += ((a >> 10) != (p >> 10)) + ((z >> 10) != (a >> 10));
}
__device__ __forceinline__ void flush_link(const LinkCount &lc, unsigned long long *ctr) {
    if (!ctr) return;
    const unsigned int sec = __reduce_add_sync(0xffffffffu, lc.sec), ln = __reduce_add_sync(0xffffffffu, lc.ln);
    if ((threadIdx.x & 31) == 0 && sec) {
        atomicAdd(&ctr[0], (unsigned long long)sec);
        atomicAdd(&ctr[1], (unsigned long long)ln);
    }
}

// One edge of a step: the bit positions of its entries in the task's arrays
// (the weights' only if they are read), whether the next lane holds the edge
// after it, and its owner's payload.  BATCH: the owner's per-source word and
// vertex instead of a value.
template <bool BATCH> struct Edge;
template <> struct Edge<false> {
    bool ok, adj;
    long long dbit, wbit;
    unsigned int pay;
};
template <> struct Edge<true> {
    bool ok, adj;
    long long dbit, wbit;
    unsigned long long pay;
    unsigned int vid;
};

// The packed entries of a lane's S edges (0 where there is none).  An entry
// that runs into the next word takes that word from the next lane when that
// lane holds the next edge (its entry then starts in that word), so a list's
// words are loaded once; only a list's or a step's last edge may load a second
// word, beside the first one's load.  Needs all 32 lanes.
template <bool WEIGHTS, int S, class E>
__device__ __forceinline__ void load_entries(const unsigned int *p, unsigned int bits, const E (&ed)[S],
                                             unsigned int (&out)[S]) {
    const unsigned int mask = 0xffffffffu >> (32 - bits);
    unsigned int lo[S], hi[S], sh[S];
#pragma unroll
    for (int q = 0; q < S; ++q) {
        const long long bit = WEIGHTS ? ed[q].wbit : ed[q].dbit;
        const unsigned int *at = p + (bit >> 5);
        sh[q] = (unsigned int)bit & 31u;
        lo[q] = ed[q].ok ? __ldg(at) : 0u;
        hi[q] = ed[q].ok && !ed[q].adj && sh[q] + bits > 32 ? __ldg(at + 1) : 0u;
    }
#pragma unroll
    for (int q = 0; q < S; ++q) {
        const unsigned int next = __shfl_down_sync(0xffffffffu, lo[q], 1);
        out[q] = __funnelshift_r(lo[q], ed[q].adj ? next : hi[q], sh[q]) & mask;
    }
}

// Run length (log2) for `total` edges over `nwarps` warps: kRun, halved down
// to one step of 32 edges while there are fewer runs than warps, so that a
// small task's edges are spread over warps instead of walked in turn.
__device__ __forceinline__ int run_shift(unsigned long long total, unsigned long long nwarps) {
    int sh = kRunShift;
    while (sh > 5 && (total >> sh) < nwarps) --sh;
    return sh;
}

// Walk run `run` (of 2^sh edges) of the task (edges [kb, ke) of the route), S
// steps of 32 edges at a time: f(ed, k) gets the lane's S edges and the route
// edge of the first, its others being 32 apart.  An inconsistent list is
// recorded in la.err and skipped.
template <int S, bool BATCH, bool WEIGHTS, class F>
__device__ __forceinline__ void walk_run(const ListArrays &la, const RouteView &rv, const RelaxTask &t,
                                         unsigned long long run, int sh, unsigned long long kb,
                                         unsigned long long ke, LinkCount &lc, F &&f) {
    const int lane = threadIdx.x & 31;
    const unsigned long long start = run << sh, end = (run + 1) << sh, tile = start / kTile;
    const unsigned long long k0 = start > kb ? start : kb;
    const int n = (int)((end < ke ? end : ke) - k0);
    // entries of the tile: from the owner of its first edge (or of the task's)
    // to the owner of the next tile's
    unsigned long long i = tile * kTile >= kb ? la.tile_first[rv.tbase + tile] : t.first_entry;
    const unsigned long long i_end =
        (tile + 1) * kTile < rv.n_edges ? (unsigned long long)la.tile_first[rv.tbase + tile + 1] + 1 : rv.n_ent;
    if (i >= i_end || i_end > rv.n_ent) {           // inconsistent tile index (warp-uniform)
        if (lane == 0) atomicOr(la.err, 1u);
        return;
    }
    if (k0 != tile * kTile && k0 != kb) {
        // the last entry that starts at or before k0, to within a window
        for (unsigned long long m = i_end - i; m > 32;) {
            const unsigned long long step = (m + 31) / 32, j = i + lane * step;
            const bool le = lane == 0 || (j < i_end && la.ebase[rv.rbase + j] <= k0);
            i += (31 - __clz(__ballot_sync(0xffffffffu, le))) * step;
            m = step < i_end - i ? step : i_end - i;
        }
    }
    long long e_prev = -1;                          // edge before the run (link counts)
    bool want_prev = t.link_ctr && k0 > kb;
    int pos = 0;
    while (pos < n) {
        // window of the entries i .. i + 31: lane 31 only marks where the
        // edges of the others end
        const bool in = i + lane < i_end;
        const unsigned long long idx = rv.rbase + (in ? i + lane : 0);
        int rel = kRun;                             // list start relative to k0
        long long delta = 0;                        // edge = k + delta
        unsigned long long pay64 = 0;
        unsigned int pay = 0, vid = 0;
        if (in) {
            const long long eb = (long long)la.ebase[idx];
            const long long d = eb - (long long)k0;
            rel = d < 0 ? -1 : d < (long long)kRun ? (int)d : kRun;
            delta = t.mode == kModeCompact ? 0 : (long long)la.soff[idx] - eb;
            if (BATCH) {
                pay64 = la.pay64[idx];
                vid = la.vid[idx];
            } else {
                pay = la.pay[idx];
            }
        }
        const int r0 = __shfl_sync(0xffffffffu, rel, 0), r31 = __shfl_sync(0xffffffffu, rel, 31);
        const int wend = r31 < n ? r31 : n;
        if (r0 > pos) {                             // the window starts past pos: an inconsistent list
            if (lane == 0) atomicOr(la.err, 1u);
            return;
        }
        if (wend <= pos) {                          // pos belongs to a later window
            i += 31;
            continue;
        }
        if (want_prev) {
            // the edge before k0: of the same list, or the last of the list before it
            want_prev = false;
            const unsigned int le = __ballot_sync(0xffffffffu, rel < 0);
            if (le) {
                e_prev = (long long)(k0 - 1) + __shfl_sync(0xffffffffu, delta, 31 - __clz(le));
            } else {                                // k0 starts the window's first list
                const unsigned long long j = rv.rbase + (i ? i - 1 : 0);
                e_prev = (long long)(k0 - 1) + ((long long)la.soff[j] - (long long)la.ebase[j]);
            }
        }
        // per list, once a window: where its entries lie (for route edge k0, had
        // it been the list's), and that its edges of this run are present
        const long long dbase = (delta + (long long)k0) * t.src.dst_bits - t.src.dst_off;
        const long long wbase = WEIGHTS ? (delta + (long long)k0) * t.src.w_bits - t.src.w_off : 0;
        {
            const int next = __shfl_down_sync(0xffffffffu, rel, 1);
            const int f = rel < 0 ? 0 : rel, z = next < n ? next : n;
            const long long e0 = delta + (long long)k0;
            if (__any_sync(0xffffffffu, lane < 31 && f < z &&
                                            (e0 + f < (long long)t.src.e_lo || e0 + z > (long long)t.src.e_hi))) {
                if (lane == 0) atomicOr(la.err, 8u);
                pos = wend;
                i += 31;
                continue;
            }
        }
        int before = __popc(__ballot_sync(0xffffffffu, rel < pos));
        for (int b0 = pos; b0 < wend; b0 += 32 * S) {
            Edge<BATCH> ed[S];
#pragma unroll
            for (int q = 0; q < S; ++q) {
                const int b = b0 + 32 * q;
                ed[q].ok = ed[q].adj = false;
                if (b >= wend) continue;            // warp-uniform
                const unsigned int at = (unsigned int)(rel - b);
                const unsigned int heads = __reduce_or_sync(0xffffffffu, at < 32u ? 1u << at : 0u);
                const int own = before + __popc(heads & (0xffffffffu >> (31 - lane))) - 1;
                before += __popc(heads);
                ed[q].dbit = __shfl_sync(0xffffffffu, dbase, own) + (unsigned int)(b + lane) * t.src.dst_bits;
                if (WEIGHTS)
                    ed[q].wbit = __shfl_sync(0xffffffffu, wbase, own) + (unsigned int)(b + lane) * t.src.w_bits;
                if constexpr (BATCH) {
                    ed[q].pay = __shfl_sync(0xffffffffu, pay64, own);
                    ed[q].vid = __shfl_sync(0xffffffffu, vid, own);
                } else {
                    ed[q].pay = __shfl_sync(0xffffffffu, pay, own);
                }
                ed[q].ok = b + lane < wend;
                ed[q].adj = lane < 31 && b + lane + 1 < wend && !((heads >> (lane + 1)) & 1u);
                if (t.link_ctr) {
                    const long long e = (long long)(k0 + b + lane) + __shfl_sync(0xffffffffu, delta, own);
                    long long p = __shfl_up_sync(0xffffffffu, e, 1);
                    if (lane == 0) p = e_prev;
                    if (ed[q].ok) {
                        count_link(lc, e, p, t.src.dst_bits);
                        if (WEIGHTS) count_link(lc, e, p, t.src.w_bits);
                    }
                    e_prev = __shfl_sync(0xffffffffu, e, min(31, wend - 1 - b));
                }
            }
            f(ed, k0 + b0 + lane);
        }
        pos = wend;
        i += 31;
    }
}

// Every run of the task, one per warp in turn.
template <int S, bool BATCH, bool WEIGHTS, class F>
__device__ __forceinline__ void walk_task(const ListArrays &la, const RouteView &rv, const RelaxTask &t,
                                          unsigned long long kb, unsigned long long ke, LinkCount &lc, F &&f) {
    if (kb >= ke) return;
    const unsigned long long nwarps = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
    const int sh = run_shift(ke - kb, nwarps);
    const unsigned long long last = (ke - 1) >> sh;
    for (unsigned long long run = (kb >> sh) + ((blockIdx.x * blockDim.x + threadIdx.x) >> 5); run <= last;
         run += nwarps)
        walk_run<S, BATCH, WEIGHTS>(la, rv, t, run, sh, kb, ke, lc, f);
}

// Place a block's list entries: every thread of the block calls it, each warp
// with its own (warp-uniform) numbers of entries and edges.  One atomic per
// block on the packed cursor; returns the warp's first entry and edge.
struct ListPlace {
    unsigned long long entry, edge;
};
__device__ __forceinline__ ListPlace block_reserve(unsigned int n_ent, unsigned long long n_edges,
                                                   unsigned long long *cursor, unsigned long long &total_edges) {
    __shared__ unsigned long long s_own[kRelaxBlock / 32], s_base;
    const int wid = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) s_own[wid] = (n_edges << 30) + n_ent;
    __syncthreads();
    unsigned long long before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kRelaxBlock / 32; ++w) {
        const unsigned long long x = s_own[w];
        before += w < wid ? x : 0ull;
        all += x;
    }
    if (threadIdx.x == 0) s_base = all ? atomicAdd(cursor, all) : 0ull;
    __syncthreads();
    const unsigned long long at = s_base + before;
    total_edges = all >> 30;
    __syncthreads();                                // the shared words are free again
    return {at & kSpEntries, at >> 30};
}

// Blocks of a launch over route edges [kb, ke): a warp per step of 32 edges,
// at most `cap` (the runs then grow, see run_shift).
inline unsigned int run_blocks(unsigned long long kb, unsigned long long ke, unsigned int cap) {
    const unsigned long long runs = (ke - 1) / 32 - kb / 32 + 1;
    const unsigned long long blocks = (runs + kRelaxBlock / 32 - 1) / (kRelaxBlock / 32);
    return blocks < cap ? (unsigned int)blocks : cap;
}

// The push of a second pass: its list, from the range's resident copy.
inline RelaxTask sp_push_task(const SecondPassRange &r) {
    RelaxTask t{};
    t.mode = kModeDevice;
    t.src = r.src;
    t.device_sized = true;
    t.sp_cursor = r.cursor;
    t.sp_rbase = r.vlo;
    t.sp_tbase = r.tbase;
    return t;
}

// Blocks of a take, in at most one resident wave.
inline unsigned int sp_take_blocks(unsigned long long vertices, unsigned int per_block) {
    const unsigned long long cap = 8ull * device_sms(), n = (vertices + per_block - 1) / per_block;
    return (unsigned int)(n < cap ? n : cap);
}

}  // namespace hytg
