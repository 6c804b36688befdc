// Batched runs: up to 64 BFS or SSSP sources, or up to 32 personalised
// PageRank seeds, share one run and therefore every partition transfer.  The
// planner works on the union frontier (bit v set when v is active for any
// source), so each partition's edges cross the host link once per iteration
// for all sources together.
//
// Per-vertex state (values in frames of 8 sources, see BatchState):
//   BFS/SSSP  fr[v], vis[v], nxt[v]  64-bit source masks (frontier, reached,
//             reached or improved this iteration); *bval(v, s) level or
//             distance of source s.
//   PPR       *bdelta(v, s), *brank(v, s), *bmsg(v, s) (the push of seed s
//             taken this iteration), fr32[v] mask of seeds taken.
#include "common.cuh"
#include "edge_runs.cuh"

namespace hytg {

namespace {

inline unsigned int grid_for(unsigned long long n, unsigned int block) {
    unsigned long long g = (n + block - 1) / block;
    const unsigned long long cap = 32ull * device_sms();
    if (g > cap) g = cap;
    return g == 0 ? 1u : (unsigned int)g;
}

__global__ void k_frame_init(BatchState b, unsigned long long V, unsigned int g) {
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    const unsigned long long t0 = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    const unsigned long long n = V * kFrameSources;
    if (b.mode == kBatchPPR) {
        // messages too: the vector push adds a whole frame's messages
        for (unsigned long long i = t0; i < n; i += stride) {
            b.delta[g][i] = 0.0f;
            b.rank[g][i] = 0.0f;
            b.msg[g][i] = 0.0f;
        }
    } else {
        for (unsigned long long i = t0; i < n; i += stride) b.val[g][i] = 0xFFFFFFFFu;
    }
}

// Masks and bitmap of a new run (the frames are filled by k_frame_init).
__global__ void k_b_init(BatchState b, unsigned long long V, unsigned long long n_words_alloc,
                         unsigned int *bm) {
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    const unsigned long long t0 = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    if (b.mode == kBatchPPR) {
        for (unsigned long long v = t0; v < V; v += stride) b.fr32[v] = 0;
        for (unsigned long long i = t0; i < kBatchHubCopies * b.n_hub * kMaxPprSeeds; i += stride) b.hub[i] = 0.0f;
    } else {
        for (unsigned long long v = t0; v < V; v += stride) {
            b.fr[v] = 0;
            b.vis[v] = 0;
            b.nxt[v] = 0;
        }
    }
    for (unsigned long long w = t0; w < n_words_alloc; w += stride) bm[w] = 0;
}

// Sources (internal ids) enter the frontier.  One thread per source.
__global__ void k_b_sources(BatchState b, const unsigned int *src, unsigned int K, float base,
                            unsigned int *bm) {
    const unsigned int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= K) return;
    const unsigned int v = src[s];
    if (b.mode == kBatchPPR) {
        *bdelta(b, v, s) = base;
    } else {
        atomicOr(&b.fr[v], 1ull << s);
        atomicOr(&b.vis[v], 1ull << s);
        *bval(b, v, s) = 0u;
    }
    atomicOr(&bm[v >> 5], 1u << (v & 31));
}

// BFS/SSSP after an iteration: the improved sources of v become its frontier.
// BFS also records the level of each newly reached source.  One warp per 32
// vertices so the bitmap word is written whole (the binning pass cleared it).
__global__ void k_b_commit(BatchState b, unsigned long long V, unsigned long long n_words_alloc,
                           unsigned int level, unsigned int *bm) {
    if (b.loop) level = b.loop->it;
    const int lane = threadIdx.x & 31;
    const unsigned long long nw = (unsigned long long)gridDim.x * (blockDim.x >> 5);
    for (unsigned long long w = (blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) >> 5;
         w < n_words_alloc; w += nw) {
        const unsigned long long v = w * 32 + lane;
        unsigned long long n = 0;
        if (v < V) {
            n = b.nxt[v];
            if (b.mode == kBatchBFS && n) {
                n &= ~b.vis[v];
                b.vis[v] |= n;
                unsigned long long m = n;
                while (m) {
                    const int s = __ffsll((long long)m) - 1;
                    m &= m - 1;
                    *bval(b, v, (unsigned int)s) = level;
                }
            }
            b.fr[v] = n;
            if (b.nxt[v]) b.nxt[v] = 0;
        }
        const unsigned int word = __ballot_sync(0xffffffffu, n != 0);
        if (lane == 0) bm[w] = word;
        if (b.alive && word) {
            unsigned long long orv = n;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) orv |= __shfl_xor_sync(0xffffffffu, orv, o);
            if (lane == 0) atomicOr(b.alive, orv);
        }
    }
}

// PPR: the hub copies' sums enter the residuals (ppr_edges).  A thread per hub
// id and seed; pushes and other folds may run meanwhile, so a copy is swapped
// out.  The sixteen loads are in flight together, and copies without pushes
// are left alone.
__global__ void k_b_hub_fold(BatchState b) {
    const unsigned int i = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned int v = i / kMaxPprSeeds, s = i % kMaxPprSeeds;
    if (v >= b.n_hub || b.delta[s / kFrameSources] == nullptr) return;
    float x[kBatchHubCopies];
#pragma unroll
    for (unsigned int r = 0; r < kBatchHubCopies; ++r) x[r] = __ldcg(b_hub(b, r, v, s));
    double sum = 0.0;
#pragma unroll
    for (unsigned int r = 0; r < kBatchHubCopies; ++r)
        if (x[r] != 0.0f) sum += (double)atomicExch(b_hub(b, r, v, s), 0.0f);
    if (sum != 0.0) atomicAdd(bdelta(b, v, s), (float)sum);
}
cudaError_t hub_fold(const BatchState &b, cudaStream_t s) {
    if (b.n_hub) k_b_hub_fold<<<(b.n_hub * kMaxPprSeeds + 255) / 256, 256, 0, s>>>(b);
    return cudaGetLastError();
}

// PPR: for every vertex marked in the bitmap, take the residual of each seed
// above eps (rank += delta, delta = 0, msg = d * delta / D_o) and keep the
// vertex in the frontier iff some seed was taken.  One warp per bitmap word,
// lanes are seeds.
__global__ void k_b_take(BatchState b, const unsigned long long *off, unsigned long long n_words_alloc,
                         unsigned int K, float damping, float eps, unsigned int *bm) {
    const int lane = threadIdx.x & 31;
    const unsigned long long nw = (unsigned long long)gridDim.x * (blockDim.x >> 5);
    for (unsigned long long w = (blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) >> 5;
         w < n_words_alloc; w += nw) {
        unsigned int bits = bm[w];
        if (bits == 0) continue;
        unsigned int keep = 0;
        unsigned int seen = 0;
        while (bits) {
            const int bit = __ffs(bits) - 1;
            bits &= bits - 1;
            const unsigned long long v = w * 32 + bit;
            const unsigned long long deg = off[v + 1] - off[v];
            // lanes are seeds; a seed past K, or in a frame not allocated, has no state
            const bool has = lane < (int)K && b.delta[lane >> 3] != nullptr;
            const float dl = has ? *bdelta(b, v, lane) : 0.0f;
            const bool act = has && dl > eps;
            float msg = 0.0f;
            if (act) {
                *bdelta(b, v, lane) = 0.0f;
                *brank(b, v, lane) += dl;
                msg = deg ? damping * dl / (float)deg : 0.0f;
            }
            if (has) *bmsg(b, v, lane) = msg;
            const unsigned int mask = __ballot_sync(0xffffffffu, act);
            if (lane == 0) b.fr32[v] = mask;
            if (mask) keep |= 1u << bit;
            seen |= mask;
        }
        if (lane == 0) {
            bm[w] = keep;
            if (b.alive && seen) atomicOr(b.alive, (unsigned long long)seen);
        }
    }
}

// Serving: clear one slot's column, then seed its source (at an iteration
// boundary: no relax of the slot is in flight, and the slot's source enters
// through nxt / delta so that the next commit or take activates it).
__global__ void k_serve_clear(BatchState b, unsigned long long V, unsigned int slot) {
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    const unsigned long long bit = 1ull << slot;
    for (unsigned long long v = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; v < V;
         v += stride) {
        if (b.mode == kBatchPPR) {
            *bdelta(b, v, slot) = 0.0f;
            *brank(b, v, slot) = 0.0f;
        } else {
            *bval(b, v, slot) = 0xFFFFFFFFu;
            if (b.fr[v] & bit) b.fr[v] &= ~bit;
            if (b.vis[v] & bit) b.vis[v] &= ~bit;
            if (b.nxt[v] & bit) b.nxt[v] &= ~bit;
        }
    }
}
__global__ void k_serve_seed(BatchState b, unsigned int slot, unsigned int src, float base,
                             unsigned int *bm) {
    if (b.mode == kBatchPPR) {
        *bdelta(b, src, slot) = base;
        atomicOr(&bm[src >> 5], 1u << (src & 31));
    } else {
        if (b.mode == kBatchSSSP) *bval(b, src, slot) = 0u;
        atomicOr(&b.nxt[src], 1ull << slot);
    }
}

// One finished slot's result in original vertex order: BFS levels relative to
// the slot's admission iteration, SSSP distances, PPR ranks normalised.
__global__ void k_serve_extract(BatchState b, unsigned long long V, unsigned int slot,
                                const unsigned int *perm, unsigned int offset, void *out,
                                const double *sums) {
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long v = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; v < V;
         v += stride) {
        const unsigned long long ov = perm ? perm[v] : v;
        if (b.mode == kBatchPPR) {
            const double S = sums[slot];
            ((float *)out)[ov] = S > 0.0 ? (float)((double)*brank(b, v, slot) / S) : 0.0f;
        } else {
            const unsigned int x = *bval(b, v, slot);
            ((unsigned int *)out)[ov] = (x == 0xFFFFFFFFu || b.mode != kBatchBFS) ? x : x - offset;
        }
    }
}

// Multi-source BFS relax: one lane per edge; the sources of u not yet
// reached at v are ORed into nxt[v].
constexpr int kBatchSteps = 4;
__global__ void __launch_bounds__(kRelaxBlock) k_relax_msbfs(BatchState b, ListArrays la,
                                                             const Summary *sum, RelaxTask t) {
    if (b.loop && !b.loop->work) return;
    unsigned long long kb, ke;
    const RouteView rv = task_view(t, sum, kb, ke);
    LinkCount lc;
    walk_task<kBatchSteps, true, false>(la, rv, t, kb, ke, lc, [&](const Edge<true> (&ed)[kBatchSteps], unsigned long long) {
        unsigned int dv[kBatchSteps];
        unsigned long long seen[kBatchSteps];
        load_entries<false>(t.src.dst, t.src.dst_bits, ed, dv);
        // reached before, or marked by another edge of this iteration: a hub's
        // word would otherwise take an atomic from every edge that ends there
#pragma unroll
        for (int q = 0; q < kBatchSteps; ++q)
            seen[q] = ed[q].ok ? __ldcg(&b.vis[dv[q]]) | __ldcg(&b.nxt[dv[q]]) : ~0ull;
#pragma unroll
        for (int q = 0; q < kBatchSteps; ++q) {
            const unsigned long long nb = ed[q].pay & ~seen[q];
            if (ed[q].ok && nb) atomicOr(&b.nxt[dv[q]], nb);
        }
    });
    flush_link(lc, t.link_ctr);
}

// Multi-source SSSP and batched PPR relax.  A warp loads 32 edges at once
// (coalesced), one per lane, each with its source vertex u and the mask of
// sources active at u.  PPR: ppr_edges.  SSSP: when the masks
// are dense (on average "batch_sparse_below" or more sources per edge) the
// warp walks its edges one at a time with a lane per source (s = lane and
// lane + 32), reading each source's value row in one sector per frame;
// otherwise every lane keeps its own edge and loops over the sources active
// at its u, so that 32 edges' loads are in flight together instead of one
// edge's.
__device__ __forceinline__ void mssssp_edges(const BatchState &b, unsigned int v, unsigned int w, unsigned int u,
                                             unsigned long long f, unsigned int *overflow) {
    const int lane = threadIdx.x & 31;
    const unsigned int pop = __reduce_add_sync(0xffffffffu, (unsigned int)__popcll(f));
    if (pop < b.sparse_below * 32u) {
        // sparse masks: a lane per edge, looping over its active sources
        unsigned long long imp = 0;
        while (f) {
            const unsigned int s = (unsigned int)(__ffsll((long long)f) - 1);
            f &= f - 1;
            const unsigned long long nd = (unsigned long long)__ldcg(bval(b, u, s)) + w;
            if (nd >= 0xFFFFFFFEull) {
                *overflow = 1u;
            } else if ((unsigned int)nd < __ldcg(bval(b, v, s))) {
                atomicMin(bval(b, v, s), (unsigned int)nd);
                imp |= 1ull << s;
            }
        }
        if (imp) atomicOr(&b.nxt[v], imp);
        return;
    }
    unsigned int todo = __ballot_sync(0xffffffffu, f != 0);
    while (todo) {
        const int jj = __ffs(todo) - 1;
        todo &= todo - 1;
        const unsigned int vj = __shfl_sync(0xffffffffu, v, jj), uj = __shfl_sync(0xffffffffu, u, jj);
        const unsigned int wj = __shfl_sync(0xffffffffu, w, jj);
        const unsigned long long fj = __shfl_sync(0xffffffffu, f, jj);
        unsigned long long imp = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const unsigned int s = lane + 32 * h;
            bool better = false;
            if ((fj >> s) & 1ull) {
                const unsigned long long nd = (unsigned long long)__ldcg(bval(b, uj, s)) + wj;
                if (nd >= 0xFFFFFFFEull) {
                    *overflow = 1u;
                } else if ((unsigned int)nd < __ldcg(bval(b, vj, s))) {
                    atomicMin(bval(b, vj, s), (unsigned int)nd);
                    better = true;
                }
            }
            imp |= (unsigned long long)__ballot_sync(0xffffffffu, better) << (32 * h);
        }
        if (lane == 0 && imp) atomicOr(&b.nxt[vj], imp);
    }
}

// PPR push of 32 edges, one per lane: u's messages for the seeds in m to w's
// residuals.  Eight lanes share an edge, each with four seeds (a 16-byte half
// of a frame's sector), so a warp has four edges in flight per load and per
// vector reduction; a lane that walked its own edge's eight halves waited for
// each load in turn.  The other seeds of a half carry a zero message (the take
// kernels write 0 for every seed they do not take), so adding them leaves
// their residuals unchanged; a half with no active seed is skipped.
//
// w's frontier bit is looked at before it is set: with R-MAT's in-degree skew
// 15 % of the edges of a 2^18-vertex graph end in the first 32 vertices, one
// word, and as many atomics on one address took most of the relax's time.
// Both together: 590 K edges with 32 seeds each, 260 -> 70 us (70 G vector
// reductions/s).
//
// Pushes to the lowest ids go to one of sixteen copies of their rows, folded
// before every take that looks at them.  The copies are for the rounding: a hub
// that 10^5 equal messages reach in one iteration gathers a bias of 4e-5 in
// one 32-bit sum (Chung-Lu 2.1, 4 M edges, resident: result off by 1.1e-5 in
// the 2-norm), and sixteen sums of a sixteenth are each that much closer
// (9.7e-7).  The same graph's run went from 69 to 40 ms, since one address no
// longer takes 3 % of all pushes; R-MAT 18, whose targets are flatter, pays 3 %
// for the test and the folds.
// (The plain load may miss a bit set meanwhile, never see one too many: bits
// are only cleared between relaxes, by earlier kernels of the main stream.)
__device__ __forceinline__ void ppr_edges(const BatchState &b, unsigned int w, unsigned int u, unsigned int m,
                                          unsigned int *bm) {
    const int lane = threadIdx.x & 31, part = lane & 7, sub = lane >> 3;
    const unsigned int copy = sm_id() % kBatchHubCopies;
    if (m && !((bm[w >> 5] >> (w & 31)) & 1u)) atomicOr(&bm[w >> 5], 1u << (w & 31));
    constexpr int kTurns = 4;                       // 16 edges' messages in flight
#pragma unroll
    for (int i0 = 0; i0 < 8; i0 += kTurns) {
        float4 x[kTurns];
        float *to[kTurns];
#pragma unroll
        for (int i = 0; i < kTurns; ++i) {
            const int e = (i0 + i) * 4 + sub;
            const unsigned int we = __shfl_sync(0xffffffffu, w, e), ue = __shfl_sync(0xffffffffu, u, e);
            const unsigned int me = __shfl_sync(0xffffffffu, m, e);
            to[i] = nullptr;
            if ((me >> (4 * part)) & 0xFu) {
                const unsigned int g = part >> 1, h = 4 * (part & 1);
                x[i] = __ldcg((const float4 *)(b.msg[g] + (unsigned long long)ue * kFrameSources + h));
                to[i] = we < b.n_hub ? b_hub(b, copy, we, 4 * part)
                                     : b.delta[g] + (unsigned long long)we * kFrameSources + h;
            }
        }
#pragma unroll
        for (int i = 0; i < kTurns; ++i)
            if (to[i]) atomicAdd((float4 *)to[i], x[i]);
    }
}

template <int MODE>
__global__ void __launch_bounds__(kRelaxBlock) k_relax_mswarp(BatchState b, ListArrays la,
                                                              const Summary *sum, RelaxTask t,
                                                              unsigned int *bm,
                                                              unsigned int *overflow) {
    if (b.loop && !b.loop->work) return;
    unsigned long long kb, ke;
    const RouteView rv = task_view(t, sum, kb, ke);
    LinkCount lc;
    walk_task<kBatchSteps, true, MODE == kBatchSSSP>(la, rv, t, kb, ke, lc, [&](const Edge<true> (&ed)[kBatchSteps], unsigned long long) {
        unsigned int dv[kBatchSteps], wv[kBatchSteps] = {};
        load_entries<false>(t.src.dst, t.src.dst_bits, ed, dv);
        if (MODE == kBatchSSSP) load_entries<true>(t.src.w, t.src.w_bits, ed, wv);
#pragma unroll
        for (int q = 0; q < kBatchSteps; ++q) {
            const unsigned long long f = ed[q].ok ? ed[q].pay : 0ull;
            if (!__any_sync(0xffffffffu, f != 0)) continue;
            if (MODE == kBatchPPR) ppr_edges(b, dv[q], ed[q].vid, (unsigned int)f, bm);
            else mssssp_edges(b, dv[q], wv[q], ed[q].vid, f, overflow);
        }
    });
    flush_link(lc, t.link_ctr);
}

// Batched PPR second pass over a resident range [vlo, vhi) (Sec. VI-A): the
// seeds whose residual at a vertex of the range rose above eps during this
// iteration are taken again, the vertices listed with their masks of taken
// seeds, and k_relax_mswarp pushes the list from the resident copy.  A warp
// takes 32 consecutive vertices, lanes are seeds; eight vertices' residuals
// are read together (one at a time, each waited for the one before: a
// dependent read of 128 bytes per vertex).  The residual is read and then
// subtracted with a reduction, so pushes that land meanwhile (other streams'
// relaxes) stay for later.
__global__ void __launch_bounds__(kRelaxBlock) k_bsp_take(BatchState b, const unsigned long long *off,
                                                          SecondPassRange r, ListArrays la, unsigned int K,
                                                          float damping, float eps) {
    if (b.loop && !b.loop->work) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned int lt_mask = (1u << lane) - 1u;
    const bool has = lane < (int)K && b.delta[lane >> 3] != nullptr;
    unsigned long long done = 0;
    for (unsigned long long b0 = r.vlo + blockIdx.x * (unsigned long long)kRelaxBlock; b0 < r.vhi;
         b0 += gridDim.x * (unsigned long long)kRelaxBlock) {
        const unsigned long long base = b0 + 32ull * wid, v = base + lane;
        unsigned long long o0 = 0, deg = 0;
        if (v < r.vhi) {
            o0 = off[v];
            deg = off[v + 1] - o0;
        }
        unsigned int mine = 0;                      // seeds taken at this lane's vertex
#pragma unroll
        for (int g = 0; g < 32; g += 8) {
            float dl[8];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                dl[q] = has && base + g + q < r.vhi ? __ldcg(bdelta(b, base + g + q, lane)) : 0.0f;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const bool act = dl[q] > eps;
                const unsigned int seeds = __ballot_sync(0xffffffffu, act);
                if (seeds == 0) continue;           // warp-uniform
                const unsigned long long u = base + g + q, du = __shfl_sync(0xffffffffu, deg, g + q);
                if (act) {
                    atomicAdd(bdelta(b, u, lane), -dl[q]);
                    *brank(b, u, lane) += dl[q];
                }
                if (du == 0) continue;
                // the vector push adds whole frames: the seeds not taken carry 0
                // (this task's relax of u, the only reader of u's old messages,
                // has finished on this stream)
                if (has) *bmsg(b, u, lane) = act ? damping * dl[q] / (float)du : 0.0f;
                if (lane == g + q) mine = seeds;
            }
        }
        done += (unsigned long long)__popc(mine) * deg;
        const unsigned long long d = mine ? deg : 0ull, incl = warp_scan_u64(d);
        const unsigned int bal = __ballot_sync(0xffffffffu, d > 0);
        unsigned long long block_edges;
        const ListPlace at = block_reserve(__popc(bal), __shfl_sync(0xffffffffu, incl, 31), r.cursor, block_edges);
        if (d) {
            const unsigned long long idx = at.entry + __popc(bal & lt_mask), eb = at.edge + incl - d;
            const unsigned long long t1 = (eb + d - 1) / kTile;
            if (idx >= r.vhi - r.vlo || r.tbase + t1 >= la.cap_tiles) {
                atomicOr(la.err, 16u);
            } else {
                la.ebase[r.vlo + idx] = eb;
                la.soff[r.vlo + idx] = o0;
                la.pay64[r.vlo + idx] = mine;
                la.vid[r.vlo + idx] = (unsigned int)v;
                for (unsigned long long t = (eb + kTile - 1) / kTile; t <= t1; ++t)
                    la.tile_first[r.tbase + t] = (unsigned int)idx;
            }
        }
    }
    done = warp_sum_u64(done);
    if (lane == 0 && done) atomicAdd(r.edges_out, done);
}

__global__ void k_b_out(BatchState b, unsigned long long V, unsigned int K, const unsigned int *perm,
                        unsigned int *out) {
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < V * K;
         i += stride) {
        const unsigned long long s = i / V, v = i % V;
        const unsigned long long ov = perm ? perm[v] : v;
        out[s * V + ov] = *bval(b, v, (unsigned int)s);
    }
}

__global__ void k_b_pr_sums(BatchState b, unsigned long long V, unsigned int K, double *sums) {
    const int lane = threadIdx.x & 31;
    const unsigned long long nw = (unsigned long long)gridDim.x * (blockDim.x >> 5);
    double acc = 0.0, res = 0.0;
    const bool has = lane < (int)K && b.rank[lane >> 3] != nullptr;
    for (unsigned long long v = (blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) >> 5;
         has && v < V; v += nw) {
        acc += *brank(b, v, lane);
        res += fabs((double)*bdelta(b, v, lane));
    }
    if (has) {
        atomicAdd(&sums[lane], acc);
        atomicAdd(&sums[32 + lane], res);
    }
}

__global__ void k_b_pr_out(BatchState b, unsigned long long V, unsigned int K, const unsigned int *perm,
                           const double *sums, float *out) {
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < V * K;
         i += stride) {
        const unsigned long long s = i / V, v = i % V;
        const unsigned long long ov = perm ? perm[v] : v;
        const double S = sums[s];
        out[s * V + ov] = S > 0.0 ? (float)((double)*brank(b, v, (unsigned int)s) / S) : 0.0f;
    }
}

}  // namespace

cudaError_t launch_b_init(const BatchState &b, unsigned long long V, unsigned long long n_words_alloc,
                          const unsigned int *src_dev, unsigned int K, float base, unsigned int *bm,
                          cudaStream_t s) {
    k_b_init<<<grid_for(V, 256), 256, 0, s>>>(b, V, n_words_alloc, bm);
    if (K) k_b_sources<<<1, 64, 0, s>>>(b, src_dev, K, base, bm);
    return cudaGetLastError();
}

cudaError_t launch_frame_init(const BatchState &b, unsigned long long V, unsigned int g, cudaStream_t s) {
    const bool ok = b.mode == kBatchPPR ? (g < kMaxPprFrames && b.delta[g] && b.rank[g])
                                        : (g < kMaxFrames && b.val[g]);
    if (!ok) return cudaErrorInvalidValue;
    k_frame_init<<<grid_for(V * kFrameSources, 256), 256, 0, s>>>(b, V, g);
    return cudaGetLastError();
}

cudaError_t launch_b_commit(const BatchState &b, unsigned long long V, unsigned long long n_words_alloc,
                            unsigned int level, unsigned int *bm, cudaStream_t s) {
    k_b_commit<<<grid_for(n_words_alloc * 32, 256), 256, 0, s>>>(b, V, n_words_alloc, level, bm);
    return cudaGetLastError();
}

cudaError_t launch_b_take(const BatchState &b, const unsigned long long *off,
                          unsigned long long n_words_alloc, unsigned int K, float damping, float eps,
                          unsigned int *bm, cudaStream_t s) {
    cudaError_t e = hub_fold(b, s);
    if (e != cudaSuccess) return e;
    k_b_take<<<grid_for(n_words_alloc * 32, 256), 256, 0, s>>>(b, off, n_words_alloc, K, damping, eps, bm);
    return cudaGetLastError();
}

cudaError_t launch_relax_batched(const BatchState &b, const ListArrays &la, const Summary *sum,
                                 const RelaxTask &t, int grid_cap, unsigned int *bm,
                                 unsigned int *overflow, cudaStream_t s) {
    unsigned int grid = (unsigned int)grid_cap;
    if (!t.device_sized && !t.dev_edge) {
        if (t.k_begin >= t.k_end) return t.sp_reset ? cudaMemsetAsync(t.sp_reset, 0, 8, s) : cudaSuccess;
        grid = run_blocks(t.k_begin, t.k_end, grid);
    }
    if (b.mode == kBatchBFS) k_relax_msbfs<<<grid, kRelaxBlock, 0, s>>>(b, la, sum, t);
    else if (b.mode == kBatchSSSP)
        k_relax_mswarp<kBatchSSSP><<<grid, kRelaxBlock, 0, s>>>(b, la, sum, t, bm, overflow);
    else k_relax_mswarp<kBatchPPR><<<grid, kRelaxBlock, 0, s>>>(b, la, sum, t, bm, overflow);
    return cudaGetLastError();
}

cudaError_t launch_second_pass_batched(const BatchState &b, const unsigned long long *off,
                                       const SecondPassRange &r, const ListArrays &la, const Summary *sum,
                                       unsigned int K, float damping, float eps, unsigned int *bm,
                                       cudaStream_t s) {
    if (r.vhi <= r.vlo) return cudaSuccess;
    if ((r.vlo & 31) || b.mode != kBatchPPR || r.vhi - r.vlo > kSpEntries || r.E1 - r.E0 > kSpEdgesMax)
        return cudaErrorInvalidValue;
    cudaError_t e = r.vlo < b.n_hub ? hub_fold(b, s) : cudaSuccess;
    if (e != cudaSuccess) return e;
    k_bsp_take<<<sp_take_blocks(r.vhi - r.vlo, kRelaxBlock), kRelaxBlock, 0, s>>>(b, off, r, la, K, damping, eps);
    return launch_relax_batched(b, la, sum, sp_push_task(r),
                                r.E1 > r.E0 ? (int)run_blocks(0, r.E1 - r.E0, 8 * device_sms()) : 1, bm, nullptr, s);
}

cudaError_t launch_serve_admit(const BatchState &b, unsigned long long V, unsigned int slot,
                               unsigned int src, float base, unsigned int *bm, cudaStream_t s) {
    k_serve_clear<<<grid_for(V, 256), 256, 0, s>>>(b, V, slot);
    k_serve_seed<<<1, 1, 0, s>>>(b, slot, src, base, bm);
    return cudaGetLastError();
}

cudaError_t launch_serve_extract(const BatchState &b, unsigned long long V, unsigned int slot,
                                 const unsigned int *perm, unsigned int offset, void *out,
                                 double *sums, cudaStream_t s) {
    if (b.mode == kBatchPPR) {
        cudaError_t e = cudaMemsetAsync(sums, 0, 64 * sizeof(double), s);
        if (e != cudaSuccess) return e;
        k_b_pr_sums<<<grid_for(V * 32, 256), 256, 0, s>>>(b, V, 32, sums);
    }
    k_serve_extract<<<grid_for(V, 256), 256, 0, s>>>(b, V, slot, perm, offset, out, sums);
    return cudaGetLastError();
}

cudaError_t launch_b_finalize(const BatchState &b, unsigned long long V, unsigned int K,
                              const unsigned int *perm, void *out, double *sums, cudaStream_t s) {
    if (b.mode == kBatchPPR) {
        cudaError_t e = hub_fold(b, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(sums, 0, 64 * sizeof(double), s);
        if (e != cudaSuccess) return e;
        k_b_pr_sums<<<grid_for(V * 32, 256), 256, 0, s>>>(b, V, K, sums);
        k_b_pr_out<<<grid_for(V * K, 256), 256, 0, s>>>(b, V, K, perm, sums, (float *)out);
    } else {
        k_b_out<<<grid_for(V * K, 256), 256, 0, s>>>(b, V, K, perm, (unsigned int *)out);
    }
    return cudaGetLastError();
}

}  // namespace hytg
