// Small-frontier iterations of the device loop (BFS, SSSP, CC from one source):
// one cluster of eight blocks runs whole iterations, one after another, while
// the frontier fits one vertex per thread.
//
// On high-diameter graphs a run is thousands of iterations of a few hundred or
// thousand vertices.  The loop's graph body spends 25 to 29 us on each: five
// kernels, two walks over the whole bitmap, and the latency of each kernel's
// start and end.  Here the frontier is an explicit queue, an iteration is
//   1  a thread takes a vertex: value, row, partition; partition counts (the
//      inputs of Eq. 1-3) are summed in each block's shared memory; a warp
//      walks the edges of its 32 vertices as the relax kernels do and loads
//      the first 128 edges' targets and values;
//   -- cluster barrier --
//   2  every block reads all blocks' counts, decides the routes of all
//      partitions (a thread per partition), and whether the iteration belongs
//      here;
//   3  the warps push, and append each vertex they activate first (the bitmap
//      bit's old value) to the next queue;
//   -- cluster barrier --
// and costs two hardware barriers and one chain of dependent loads, so what
// bounds it is that latency (host memory for zero-copy edges).  Eight blocks
// are the largest portable cluster; 512 threads leave a thread registers to
// hold a step group's edges, targets and values across the first barrier.
// Measured on a 1021 x 1031 mesh (whole calls): BFS, 1,073 iterations, 27.4 ->
// 8.6 ms; SSSP, 2,036 iterations, 58 -> 19 ms (device).
//
// A partition routed to compaction is gathered here too: its few active lists
// go from host memory through the warp's registers to the push, the bytes a
// gather into the compaction buffer would move, without the buffer (unless
// host threads compact, see TailArgs::gather).
//
// The bitmap stays the truth: bits are cleared when a vertex is taken and set
// on activation, so the kernel can stop before any iteration (a route that
// needs copies, a frontier that has grown, the caps and the cancel word of the
// loop) and the graph body takes over, with the same records, counts and
// bucket steps as if it had run every iteration itself.
#include <cooperative_groups.h>

#include "common.cuh"
#include "cost_model.cuh"
#include "edge_runs.cuh"
#include "hytg.h"

namespace cg = cooperative_groups;

namespace hytg {

namespace {

constexpr int kTailBlocks = 8, kTailThreads = 512;
static_assert(kTailBlocks * kTailThreads == (int)kTailQueue, "a thread per queue entry");
// A warp's edges at most: more would be walked by one warp while others wait.
constexpr unsigned int kTailWarpEdges = 1024;
constexpr int kTailSteps = 4;

// Each block counts its own vertices; [2]: iteration parity.
struct TailShared {
    uint4 cnt[2][kTailParts];           // per partition: active | with edges << 16, edges, lines
    uint4 head[2];                      // active, pending, smallest pending value, kTail* flags
    unsigned int len[2];                // queue lengths (block 0's are the cluster's)
};
enum : unsigned int { kTailOver = 1u, kTailStop = 2u };

struct TailEdge {
    bool ok, adj;
    long long e;                        // CSR index
    unsigned int pay;
};

struct TailTotals {
    unsigned long long parts[kRoutes], entries[kRoutes], edges[kRoutes], lines[kRoutes];
};

// The packed entries of a lane's edges, each from its own array (the cache or
// the host's, both indexed from edge 0): load_entries with a pointer per edge.
template <int S>
__device__ __forceinline__ void tail_entries(const unsigned int *const (&p)[S], unsigned int bits,
                                             const TailEdge (&ed)[S], unsigned int (&out)[S]) {
    const unsigned int mask = 0xffffffffu >> (32 - bits);
    unsigned int lo[S], hi[S], sh[S];
#pragma unroll
    for (int q = 0; q < S; ++q) {
        const unsigned long long bit = ed[q].ok ? (unsigned long long)ed[q].e * bits : 0ull;
        const unsigned int *at = p[q] + (bit >> 5);
        sh[q] = (unsigned int)bit & 31u;
        lo[q] = ed[q].ok ? __ldg(at) : 0u;
        hi[q] = ed[q].ok && !ed[q].adj && sh[q] + bits > 32 ? __ldg(at + 1) : 0u;
    }
#pragma unroll
    for (int q = 0; q < S; ++q) {
        const unsigned int next = __shfl_down_sync(0xffffffffu, lo[q], 1);
        out[q] = ed[q].ok ? __funnelshift_r(lo[q], ed[q].adj ? next : hi[q], sh[q]) & mask : 0u;
    }
}

template <int ALGO>
__global__ void __cluster_dims__(kTailBlocks, 1, 1) __launch_bounds__(kTailThreads, 1) k_tail(TailArgs a) {
    LoopCtl *ctl = a.ctl;
    if (!ctl->tail) return;                         // the same in every block
    __shared__ TailShared sh;
    __shared__ TailTotals tot;
    __shared__ unsigned int s_wb[kTailParts + 1];
    __shared__ unsigned char s_route[kTailParts];
    __shared__ unsigned char s_lane[kTailThreads];
    cg::cluster_group cl = cg::this_cluster();
    const unsigned int rank = cl.block_rank(), tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    TailShared *s0 = cl.map_shared_rank(&sh, 0);
    const unsigned int N = a.g.N;
    // queue entries go to the cluster's warps in turn, so that every warp has
    // an equal share of a small queue's vertices (and about of its edges)
    const unsigned int slot = lane * (kTailQueue / 32) + wid * kTailBlocks + rank;
    const unsigned int lt_mask = (1u << lane) - 1u;

    for (unsigned int i = tid; i < 2 * kTailParts; i += kTailThreads) ((uint4 *)sh.cnt)[i] = make_uint4(0, 0, 0, 0);
    for (unsigned int i = tid; i <= N; i += kTailThreads) s_wb[i] = a.g.part_wb[i];
    if (tid < 2) {
        sh.len[tid] = 0;
        sh.head[tid] = make_uint4(0, 0, 0xFFFFFFFFu, 0);
    }
    if (tid < kRoutes) tot.parts[tid] = tot.entries[tid] = tot.edges[tid] = tot.lines[tid] = 0;
    unsigned int it = ctl->it, bucket = ctl->bucket, n_rec = ctl->n_rec;
    const unsigned int it0 = it;
    const unsigned long long max_it = ctl->max_it;
    const unsigned int rec_cap = ctl->rec_cap;
    // running totals, kept by thread 0 of block 0
    unsigned long long t_parts[kRoutes] = {}, t_entries[kRoutes] = {}, t_edges[kRoutes] = {};
    unsigned long long t_zlines = 0, t_clines = 0, t_vertices = 0, t_alledges = 0, t_iters = 0;
    cl.sync();

    // the first queue: every set bit of the bitmap
    {
        const uint4 *bm4 = reinterpret_cast<const uint4 *>(a.st.bm_cur);
        const unsigned int n4 = (unsigned int)(a.g.n_words_alloc / 4);
        for (unsigned int i = rank * kTailThreads + tid; i < n4; i += kTailBlocks * kTailThreads) {
            const uint4 x = __ldcg(bm4 + i);
            const unsigned int w[4] = {x.x, x.y, x.z, x.w};
            const unsigned int n = __popc(x.x) + __popc(x.y) + __popc(x.z) + __popc(x.w);
            if (n == 0) continue;
            unsigned int pos = atomicAdd(&s0->len[0], n);
            for (int q = 0; q < 4; ++q)
                for (unsigned int b = w[q]; b; b &= b - 1, ++pos)
                    if (pos < kTailQueue) __stcg(&a.queue[0][pos], (i * 4 + q) * 32 + __ffs(b) - 1);
        }
    }
    cl.sync();

    LinkCount lz, lc;                               // zero-copy and compaction routes
    int cur = 0, why = kTailAgain;
    bool took = false, elig = false;
    unsigned int v = 0;
    for (;;) {
        // ---- 1: a thread takes a vertex
        const unsigned int queued = __ldcg(&a.queue[cur][slot]);
        const unsigned int n = *(volatile unsigned int *)&s0->len[cur];
        elig = false;
        if (n > kTailQueue) break;                  // grown: nothing of this iteration is taken
        unsigned int pay = 0, part = 0, deg = 0, lines = 0;
        unsigned long long o0 = 0;
        bool wait = false;                          // a later bucket's vertex
        if (slot < n) {
            v = queued;
            pay = __ldcg(&a.st.val[v]);
            o0 = a.g.off[v];
            const unsigned long long o1 = a.g.off[v + 1], d = o1 - o0;
            wait = ALGO == kSSSP && pay >= bucket && bucket != 0xFFFFFFFFu;
            elig = !wait;
            if (elig) {
                deg = d < 0x7FFFFFFull ? (unsigned int)d : 0x7FFFFFFu;
                if (deg)
                    lines = a.st.n_arrays *
                            (unsigned int)(a.m_shift >= 0
                                ? ((o1 * 4ull - 1) >> a.m_shift) - ((o0 * 4ull) >> a.m_shift) + 1
                                : lines_spanned(o0 * 4ull, d * 4ull, a.m));
                if (ALGO == kCC) {
                    // pointer jumping, as before every CC iteration
                    unsigned int l = pay;
                    for (int hop = 0; hop < 64; ++hop) {
                        const unsigned int l2 = __ldcg(&a.st.val[l]);
                        if (l2 >= l) break;
                        l = l2;
                    }
                    if (l < pay) atomicMin(&a.st.val[v], l);
                    pay = l;
                }
                atomicAnd(&a.st.bm_cur[v >> 5], ~(1u << (v & 31)));
                unsigned int lo = 0, hi = N;        // the partition of word v / 32
                while (hi - lo > 1) {
                    const unsigned int mid = (lo + hi) >> 1;
                    if (s_wb[mid] <= (v >> 5)) lo = mid; else hi = mid;
                }
                part = lo;
                uint4 *c = &sh.cnt[cur][part];
                atomicAdd(&c->x, deg ? 0x10001u : 1u);
                if (deg) {
                    atomicAdd(&c->y, deg);
                    atomicAdd(&c->z, lines);
                }
            }
        }
        if (ALGO == kSSSP) {
            // vertices of later buckets stay queued (and set in the bitmap)
            const unsigned int wm = __ballot_sync(0xffffffffu, wait);
            if (wm) {
                unsigned int pos = 0;
                const unsigned int mn = __reduce_min_sync(0xffffffffu, wait ? pay : 0xFFFFFFFFu);
                if (lane == 0) {
                    pos = atomicAdd(&s0->len[cur ^ 1], (unsigned int)__popc(wm));
                    atomicAdd(&sh.head[cur].y, (unsigned int)__popc(wm));
                    atomicMin(&sh.head[cur].z, mn);
                }
                pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(wm & lt_mask);
                if (wait && pos < kTailQueue) __stcg(&a.queue[cur ^ 1][pos], v);
            }
        }
        // the scan of the warp's edges (each lane below 2^27)
        unsigned int incl = min(deg, kTailWarpEdges + 1);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int t = __shfl_up_sync(0xffffffffu, incl, o);
            if ((int)lane >= o) incl += t;
        }
        const unsigned int total = __shfl_sync(0xffffffffu, incl, 31);
        const bool over = total > kTailWarpEdges;
        const unsigned int n_elig = __popc(__ballot_sync(0xffffffffu, elig));
        if (lane == 0 && n_elig) atomicAdd(&sh.head[cur].x, n_elig);
        if (lane == 0 && over) atomicOr(&sh.head[cur].w, (unsigned int)kTailOver);
        if (rank == 0 && tid == 0 && ctl->cancel && *ctl->cancel != 0u) atomicOr(&sh.head[cur].w, (unsigned int)kTailStop);
        // the lanes with edges, moved to the front
        const unsigned int full = over ? 0u : __ballot_sync(0xffffffffu, deg > 0);
        const unsigned int nl = __popc(full);
        if (deg > 0) s_lane[(tid & ~31u) + __popc(full & lt_mask)] = (unsigned char)lane;
        __syncwarp();
        const unsigned int from = lane < nl ? s_lane[(tid & ~31u) + lane] : lane;
        int rel = (int)__shfl_sync(0xffffffffu, incl - deg, from);
        if (lane >= nl) rel = 0x7FFFFFFF;
        const long long delta = (long long)__shfl_sync(0xffffffffu, o0, from) - rel;
        const unsigned int mypay = __shfl_sync(0xffffffffu, pay, from);
        // a resident partition's edges come from the cache unless a forced route
        // sends them over the link, as the body's gather and zero-copy relax read
        // them then
        const unsigned int mypart = __shfl_sync(0xffffffffu, part, from);     // every lane, before any condition
        const unsigned int cached =
            __ballot_sync(0xffffffffu, lane < nl && mypart < a.cp.n_cached &&
                                            (a.cp.force_route == -1 || a.cp.force_route == kRouteCache));
        // a step group's edges, targets, weights and values seen
        TailEdge ed[kTailSteps];
        int own[kTailSteps];
        unsigned int dv[kTailSteps], wv[kTailSteps] = {}, seen[kTailSteps];
        const auto load = [&](unsigned int b0) {
            const unsigned int *pd[kTailSteps], *pw[kTailSteps];
#pragma unroll
            for (int q = 0; q < kTailSteps; ++q) {
                const int b = (int)b0 + 32 * q;
                ed[q].ok = ed[q].adj = false;
                ed[q].e = 0;
                ed[q].pay = 0;
                own[q] = 0;
                pd[q] = a.host.dst;
                pw[q] = a.host.w;
                if (b >= (int)total) continue;      // warp-uniform
                const int before = __popc(__ballot_sync(0xffffffffu, rel < b));
                const unsigned int heads =
                    __reduce_or_sync(0xffffffffu, rel >= b && rel < b + 32 ? 1u << (rel - b) : 0u);
                own[q] = before + __popc(heads & (0xffffffffu >> (31 - lane))) - 1;
                ed[q].e = (long long)(b + (int)lane) + __shfl_sync(0xffffffffu, delta, own[q]);
                ed[q].pay = __shfl_sync(0xffffffffu, mypay, own[q]);
                ed[q].ok = b + (int)lane < (int)total;
                ed[q].adj = lane < 31 && b + (int)lane + 1 < (int)total && !((heads >> (lane + 1)) & 1u);
                const bool c_src = (cached >> (own[q] & 31)) & 1u;
                if (c_src) {
                    pd[q] = a.cache.dst;
                    pw[q] = a.cache.w;
                }
                const unsigned long long lim = c_src ? a.cache.e_hi : a.host.e_hi;
                if (ed[q].ok && (unsigned long long)ed[q].e >= lim) {
                    atomicOr(a.err, 8u);
                    ed[q].ok = ed[q].adj = false;
                }
            }
            tail_entries(pd, a.host.dst_bits, ed, dv);
            if (ALGO == kSSSP) tail_entries(pw, a.host.w_bits, ed, wv);
#pragma unroll
            for (int q = 0; q < kTailSteps; ++q) seen[q] = ed[q].ok ? __ldcg(&a.st.val[dv[q]]) : 0u;
        };
        const auto push = [&](unsigned int gathered) {
            bool add[kTailSteps];
#pragma unroll
            for (int q = 0; q < kTailSteps; ++q) {
                // link reads of the edges that came from host memory
                const bool c_rt = (gathered >> (own[q] & 31)) & 1u;
                const unsigned int hm =
                    __ballot_sync(0xffffffffu, ed[q].ok && !((cached >> (own[q] & 31)) & 1u));
                if (hm) {
                    const long long p = __shfl_up_sync(0xffffffffu, ed[q].e, 1);
                    const long long prev = lane > 0 && ((hm >> (lane - 1)) & 1u) ? p : -1;
                    if ((hm >> lane) & 1u) {
                        LinkCount &l = c_rt ? lc : lz;
                        count_link(l, ed[q].e, prev, a.host.dst_bits);
                        if (ALGO == kSSSP) count_link(l, ed[q].e, prev, a.host.w_bits);
                    }
                }
                unsigned int nv = ed[q].pay;
                bool ok = ed[q].ok;
                if (ALGO == kBFS) nv = ed[q].pay + 1u;
                if (ALGO == kSSSP) {
                    const unsigned long long s = (unsigned long long)ed[q].pay + wv[q];
                    if (ok && s >= 0xFFFFFFFEull) {
                        *a.st.overflow = 1u;
                        ok = false;
                    }
                    nv = (unsigned int)s;
                }
                add[q] = false;
                if (ok && nv < seen[q]) {
                    atomicMin(&a.st.val[dv[q]], nv);
                    const unsigned int bit = 1u << (dv[q] & 31);
                    add[q] = !(atomicOr(&a.st.bm_next[dv[q] >> 5], bit) & bit);
                }
            }
            unsigned int am[kTailSteps], cnt = 0;
#pragma unroll
            for (int q = 0; q < kTailSteps; ++q) {
                am[q] = __ballot_sync(0xffffffffu, add[q]);
                cnt += __popc(am[q]);
            }
            if (cnt) {
                unsigned int pos = 0;
                if (lane == 0) pos = atomicAdd(&s0->len[cur ^ 1], cnt);
                pos = __shfl_sync(0xffffffffu, pos, 0);
#pragma unroll
                for (int q = 0; q < kTailSteps; ++q) {
                    const unsigned int at = pos + __popc(am[q] & lt_mask);
                    if (add[q] && at < kTailQueue) __stcg(&a.queue[cur ^ 1][at], dv[q]);
                    pos += __popc(am[q]);
                }
            }
        };
        // the first group is on its way while the cluster meets and decides:
        // its values are those of the iteration's start either way, since
        // reductions come after the barrier
        if (full) load(0);
        cl.sync();

        // ---- 2: what this iteration is, the same in every block
        const uint4 hd = lane < kTailBlocks ? *cl.map_shared_rank(&sh.head[cur], lane)
                                            : make_uint4(0, 0, 0xFFFFFFFFu, 0);
        const unsigned int active = __reduce_add_sync(0xffffffffu, hd.x);
        const unsigned int pending = __reduce_add_sync(0xffffffffu, hd.y);
        const unsigned int pm = __reduce_min_sync(0xffffffffu, hd.z);
        const unsigned int flags = __reduce_or_sync(0xffffffffu, hd.w);
        if (active == 0) {
            if (pending == 0) {
                why = kTailDone;
                break;
            }
            // the current bucket is settled: open the next one
            unsigned long long nb = bucket > pm ? bucket : pm;
            nb += ctl->delta;
            bucket = nb < 0xFFFFFFFEull ? (unsigned int)nb : 0xFFFFFFFEu;
            if (pm >= 0xFFFFFFFEu) bucket = 0xFFFFFFFFu;
            ++it;
        } else {
            took = true;
            if ((unsigned long long)it >= max_it) {
                why = kTailMaxIt;
                break;
            }
            if (flags & kTailStop) {
                why = kTailCancel;
                break;
            }
            if ((flags & kTailOver) || n_rec >= rec_cap) break;
            bool copies = false;
            for (unsigned int i = tid; i < N; i += kTailThreads) {
                uint4 x[kTailBlocks], c = make_uint4(0, 0, 0, 0);
#pragma unroll
                for (int q = 0; q < kTailBlocks; ++q) x[q] = *cl.map_shared_rank(&sh.cnt[cur][i], q);
#pragma unroll
                for (int q = 0; q < kTailBlocks; ++q) {
                    c.x += x[q].x;
                    c.y += x[q].y;
                    c.z += x[q].z;
                }
                if (!c.y) continue;
                const int r =
                    decide_route_counts(i, a.g.part_eb[i + 1] - a.g.part_eb[i], c.x & 0xFFFFu, c.y, c.z, a.cp);
                s_route[i] = (unsigned char)r;
                copies |= r == kRouteF || (r == kRouteC && !a.gather);
                if (rank == 0) {
                    atomicAdd(&tot.parts[r], 1ull);
                    atomicAdd(&tot.entries[r], (unsigned long long)(c.x >> 16));
                    atomicAdd(&tot.edges[r], (unsigned long long)c.y);
                    atomicAdd(&tot.lines[r], (unsigned long long)c.z);
                }
            }
            if (__syncthreads_or(copies)) break;
            if (rank == 0 && tid == 0) {
                hytg_iter_record *rec = (hytg_iter_record *)ctl->rec + n_rec;
                unsigned long long parts = 0, edges = 0;
#pragma unroll
                for (int q = 1; q < kRoutes; ++q) {
                    parts += tot.parts[q];
                    edges += tot.edges[q];
                    rec->route_partitions[q] = (unsigned int)tot.parts[q];
                    rec->route_edges[q] = tot.edges[q];
                    t_parts[q] += tot.parts[q];
                    t_entries[q] += tot.entries[q];
                    t_edges[q] += tot.edges[q];
                }
                rec->route_partitions[0] = (unsigned int)(N - parts);
                rec->route_edges[0] = 0;
                t_parts[0] += N - parts;
                rec->active_vertices = active;
                rec->active_edges = edges;
                rec->f_tasks = 0;
                rec->link_bytes = (tot.lines[kRouteZ] + tot.lines[kRouteC]) * ctl->m;
                rec->device_ms = 0.0;
                t_zlines += tot.lines[kRouteZ];
                t_clines += tot.lines[kRouteC];
                t_vertices += active;
                t_alledges += edges;
                ++t_iters;
#pragma unroll
                for (int q = 0; q < kRoutes; ++q) tot.parts[q] = tot.entries[q] = tot.edges[q] = tot.lines[q] = 0;
            }
            ++n_rec;
            ++it;

            // ---- 3: the warp's edges
            if (full) {
                const unsigned int gathered = __ballot_sync(0xffffffffu, lane < nl && s_route[mypart] == kRouteC);
                push(gathered);
                for (unsigned int b0 = 32 * kTailSteps; b0 < total; b0 += 32 * kTailSteps) {
                    load(b0);
                    push(gathered);
                }
            }
        }
        took = false;
        // the other parity's counts and this queue's length were last read
        // before the barrier above and are next used after the one below
        for (unsigned int i = tid; i < N; i += kTailThreads) sh.cnt[cur ^ 1][i] = make_uint4(0, 0, 0, 0);
        if (tid == 0) {
            sh.head[cur ^ 1] = make_uint4(0, 0, 0xFFFFFFFFu, 0);
            if (rank == 0) sh.len[cur] = 0;
        }
        cl.sync();
        cur ^= 1;
    }
    // an iteration that was taken but not run goes back to the bitmap
    if (took && elig) atomicOr(&a.st.bm_cur[v >> 5], 1u << (v & 31));
    flush_link(lz, a.link_ctr + 2 * kRouteZ);
    flush_link(lc, a.link_ctr + 2 * kRouteC);
    if (rank == 0 && tid == 0) {
        for (int q = 0; q < kRoutes; ++q) {
            ctl->route_parts[q] += t_parts[q];
            ctl->route_entries[q] += t_entries[q];
            ctl->route_edges[q] += t_edges[q];
        }
        ctl->z_lines += t_zlines;
        ctl->c_lines += t_clines;
        ctl->vertices += t_vertices;
        ctl->edges += t_alledges;
        ctl->iterations += t_iters;
        ctl->n_rec = n_rec;
        ctl->it = it;
        ctl->bucket = bucket;
        // the body takes the iteration that was refused here, and a few more
        // when this launch ran none (a graph whose lists are too long for it)
        ctl->tail_not = it + (it == it0 ? 4 : 1);
        ctl->tail_its += it - it0;
        const cudaGraphConditionalHandle h = (cudaGraphConditionalHandle)a.cond;
        if (why != kTailAgain) {
            ctl->status = why == kTailDone ? kLoopDone : why == kTailMaxIt ? kLoopMaxIt : kLoopCancel;
            cudaGraphSetConditional(h, 0);
        }
    }
    cl.sync();                                      // block 0's shared memory outlives its readers
}

}  // namespace

cudaError_t launch_tail(const TailArgs &a, cudaStream_t s) {
    switch (a.st.algo) {
        case kBFS: k_tail<kBFS><<<kTailBlocks, kTailThreads, 0, s>>>(a); break;
        case kSSSP: k_tail<kSSSP><<<kTailBlocks, kTailThreads, 0, s>>>(a); break;
        case kCC: k_tail<kCC><<<kTailBlocks, kTailThreads, 0, s>>>(a); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace hytg
