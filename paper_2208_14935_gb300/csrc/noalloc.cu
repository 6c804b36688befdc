// hytg_plan_noalloc: the per-partition counting and engine selection of the
// planning kernels for a frontier that is already in device memory, for
// callers that must not allocate device memory (see include/hytg.h).  It
// keeps no scratch: partition bounds come straight from the caller's table,
// and the only intermediate sums are the caller's counts.
#include <mutex>

#include "common.cuh"
#include "cost_model.cuh"
#include "hytg.h"

namespace hytg {
namespace {

constexpr unsigned int kNaBlock = 512, kNaSpanBlock = 256;

struct NaInput {
    const unsigned int *bm;             // frontier words
    const unsigned long long *off, *vb; // row offsets, partition bounds (vertices)
    unsigned long long V;
    unsigned int n_parts, n_arrays;
    unsigned long long m;
    int m_shift;                        // log2 of m when it is a power of two, else -1
};

// Bound p of the table, clipped to V.
__device__ __forceinline__ unsigned long long na_bound(const NaInput &in, unsigned int p) {
    const unsigned long long v = in.vb[p];
    return v < in.V ? v : in.V;
}

// First word of partition p: a word belongs to the last partition that starts
// at or before it, and the first and last partition take what lies outside.
__device__ __forceinline__ unsigned long long na_word(const NaInput &in, unsigned int p) {
    return p == 0 ? 0 : p == in.n_parts ? (in.V + 31) / 32 : (na_bound(in, p) + 31) / 32;
}

__device__ __forceinline__ int na_route(const NaInput &in, unsigned int p, unsigned long long act,
                                        unsigned long long edges, unsigned long long lines, const CostParams &cp) {
    return decide_route_counts(p, in.off[na_bound(in, p + 1)] - in.off[na_bound(in, p)], act, edges, lines, cp);
}

// |A_i|, active edges and 128-byte lines (footnote to Eq. 3), per lane.
struct NaSums {
    unsigned long long act = 0, edges = 0, lines = 0;
};

// Words [w0, w0 + 4) below w_hi: a warp has their offsets in flight together.
__device__ __forceinline__ void na_count4(const NaInput &in, unsigned long long w0, unsigned long long w_hi,
                                          NaSums &t) {
    const unsigned int lane = threadIdx.x & 31;
    const unsigned long long n_words = (in.V + 31) / 32;
    unsigned int bits[4];
    unsigned long long o0[4], o1[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        bits[q] = w0 + q < w_hi ? in.bm[w0 + q] : 0u;
        if (w0 + q == n_words - 1 && (in.V & 31)) bits[q] &= (1u << (in.V & 31)) - 1u;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        o0[q] = o1[q] = 0;
        if ((bits[q] >> lane) & 1u) {
            const unsigned long long v = (w0 + q) * 32 + lane;
            o0[q] = in.off[v];
            o1[q] = in.off[v + 1];
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        t.act += (bits[q] >> lane) & 1u;
        if (o1[q] > o0[q]) {
            t.edges += o1[q] - o0[q];
            t.lines += in.n_arrays *
                       (in.m_shift >= 0 ? ((o1[q] * 4ull - 1) >> in.m_shift) - ((o0[q] * 4ull) >> in.m_shift) + 1
                                        : lines_spanned(o0[q] * 4ull, (o1[q] - o0[q]) * 4ull, in.m));
        }
    }
}

// A partition per block, 64 words a turn, counts and route in one launch.  What
// bounds a small call is launches and the chain of dependent loads: 2,048 words
// (65,536 vertices) in 72 or 300 equal partitions 5.1 / 5.9 us, half of them in
// the last one 12.3 / 11.5 us (blocks of 256: 18.5 / 16.5; of 1,024: 10.3 / 12.4).
__global__ void __launch_bounds__(kNaBlock) k_na_whole(NaInput in, CostParams cp, unsigned long long *counts,
                                                       unsigned char *routes) {
    __shared__ unsigned long long s_sum[kNaBlock / 32][3];
    const unsigned int p = blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned long long w_hi = na_word(in, p + 1);
    NaSums t;
    for (unsigned long long w0 = na_word(in, p) + wid * 4; w0 < w_hi; w0 += kNaBlock / 32 * 4)
        na_count4(in, w0, w_hi, t);
    t.act = warp_sum_u64(t.act);
    t.edges = warp_sum_u64(t.edges);
    t.lines = warp_sum_u64(t.lines);
    if (lane == 0) {
        s_sum[wid][0] = t.act;
        s_sum[wid][1] = t.edges;
        s_sum[wid][2] = t.lines;
    }
    __syncthreads();
    if (wid == 0) {
        const bool in_block = lane < kNaBlock / 32;
        const unsigned long long act = warp_sum_u64(in_block ? s_sum[lane][0] : 0ull),
                                 edges = warp_sum_u64(in_block ? s_sum[lane][1] : 0ull),
                                 lines = warp_sum_u64(in_block ? s_sum[lane][2] : 0ull);
        if (lane == 0) {
            counts[3ull * p] = act;
            counts[3ull * p + 1] = edges;
            counts[3ull * p + 2] = lines;
            routes[p] = (unsigned char)na_route(in, p, act, edges, lines, cp);
        }
    }
}

__global__ void k_na_zero(unsigned long long *counts, unsigned long long n) {
    cudaTriggerProgrammaticLaunchCompletion();
    const unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    if (i < n) counts[i] = 0ull;
}

// Equal spans of `span` words per warp, whatever the partitions: the sums of
// each partition that a span meets are added to its counts, which k_na_zero
// clears.  Its three launches overlap (programmatic dependent launch): a span
// waits for the zeros only before its first addition, and the selection's blocks
// wait, resident, for the counts: 7.7 us instead of 10.2 for the smallest call.
// Half the vertices in one partition take what equal partitions take: 2^22
// vertices in 2,048 partitions 18 / 21 us, 2^24 49 / 47 us.  (A partition per
// block, or cut into as many slices as the average partition needs, took 0.9 and
// 7.4 ms for the uneven ones.)
__global__ void __launch_bounds__(kNaSpanBlock) k_na_spans(NaInput in, unsigned long long span,
                                                           unsigned long long *counts) {
    const unsigned int lane = threadIdx.x & 31;
    const unsigned long long n_words = (in.V + 31) / 32;
    unsigned long long w = ((blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) >> 5) * span;
    cudaTriggerProgrammaticLaunchCompletion();
    if (w >= n_words) return;
    bool zeroed = false;
    const unsigned long long w_end = w + span < n_words ? w + span : n_words;
    // the last partition that starts at or before the span, 32 bounds at a time
    unsigned int p = 0;
    for (unsigned int n = in.n_parts; n > 1;) {
        const unsigned int step = (n + 31) / 32, j = p + lane * step;
        const bool le = lane == 0 || (lane * step < n && na_word(in, j) <= w);
        p += (31 - __clz(__ballot_sync(0xffffffffu, le))) * step;
        n = step < in.n_parts - p ? step : in.n_parts - p;
    }
    while (w < w_end) {                             // warp-uniform
        unsigned long long hi = na_word(in, p + 1);
        while (hi <= w) hi = na_word(in, ++p + 1);  // partitions without a word
        const unsigned long long z = hi < w_end ? hi : w_end;
        NaSums t;
        for (; w < z; w += 4) na_count4(in, w, z, t);
        w = z;
        t.act = warp_sum_u64(t.act);
        t.edges = warp_sum_u64(t.edges);
        t.lines = warp_sum_u64(t.lines);
        if (!zeroed) {                              // warp-uniform
            cudaGridDependencySynchronize();        // the counts are zero
            zeroed = true;
        }
        if (lane == 0 && t.act) {
            atomicAdd(&counts[3ull * p], t.act);
            atomicAdd(&counts[3ull * p + 1], t.edges);
            atomicAdd(&counts[3ull * p + 2], t.lines);
        }
        ++p;
    }
}

__global__ void k_na_select(NaInput in, const unsigned long long *counts, CostParams cp, unsigned char *routes) {
    const unsigned int p = blockIdx.x * blockDim.x + threadIdx.x;
    cudaGridDependencySynchronize();                // the counts are whole
    if (p < in.n_parts)
        routes[p] = (unsigned char)na_route(in, p, counts[3ull * p], counts[3ull * p + 1], counts[3ull * p + 2], cp);
}

constexpr unsigned long long kNaWholeWords = 2048, kNaSpanWords = 8;

constexpr int kNaMaxDevices = 64;
std::mutex g_na_mutex;
unsigned int g_na_sms[kNaMaxDevices] = {};

}  // namespace
}  // namespace hytg

using namespace hytg;

extern "C" hytg_status hytg_plan_noalloc(hytg_algo algo, const uint32_t *frontier,
                                         const uint64_t *offsets, uint64_t V,
                                         const uint64_t *part_vbounds, uint32_t n_parts,
                                         uint32_t n_cached, const hytg_cost_params *params,
                                         uint8_t *routes, uint64_t *counts, void *stream) {
    const int a = (int)algo;
    if (a < 0 || a > 4 || !frontier || !offsets || !part_vbounds || !routes || !counts)
        return HYTG_ERR_ARG;
    if (V == 0 || V > 0xFFFFFFFFull) return HYTG_ERR_ARG;
    if (n_parts == 0 || n_parts > HYTG_NOALLOC_MAX_PARTS || n_cached > n_parts) return HYTG_ERR_ARG;
    hytg_cost_params prm = {0.8, 0.4, 0.625, 128, 256};
    if (params) prm = *params;
    if (prm.m == 0 || prm.MR == 0 || !(prm.gamma >= 0 && prm.gamma <= 1) || !(prm.alpha >= 0) ||
        !(prm.beta >= 0) || prm.alpha > 1000 || prm.beta > 1000)
        return HYTG_ERR_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNaMaxDevices) return HYTG_ERR_CUDA;
    // an error left pending by earlier, unrelated work is not this call's to
    // report or to clear: queue nothing and leave it for its owner
    if (cudaPeekAtLastError() != cudaSuccess) return HYTG_ERR_CUDA;
    unsigned int sms = 0;
    {
        // the SM count that sizes the grid, once per device
        std::lock_guard<std::mutex> lock(g_na_mutex);
        if (!g_na_sms[dev]) {
            int n = 0;
            if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
                cudaGetLastError();
                return HYTG_ERR_CUDA;
            }
            g_na_sms[dev] = (unsigned int)n;
        }
        sms = g_na_sms[dev];
    }
    CostParams cp;
    auto q = [](double x) { return (unsigned long long)((x * (double)kParamDen) + 0.5); };
    cp.alpha_num = q(prm.alpha);
    cp.beta_num = q(prm.beta);
    cp.gamma_num = q(prm.gamma);
    cp.m = prm.m;
    cp.MR = prm.MR;
    cp.d1 = (a == kSSSP) ? 8 : 4;
    cp.d2 = 8;
    cp.n_cached = n_cached;
    cp.force_route = -1;
    cp.seed = 0;
    cp.iteration = 0;
    cudaStream_t s = (cudaStream_t)stream;
    NaInput in;
    in.bm = frontier;
    in.off = (const unsigned long long *)offsets;
    in.vb = (const unsigned long long *)part_vbounds;
    in.V = V;
    in.n_parts = n_parts;
    in.n_arrays = a == kSSSP ? 2u : 1u;
    in.m = prm.m;
    in.m_shift = log2_exact(prm.m);
    const unsigned long long n_words = (V + 31) / 32;
    unsigned long long *cnt = (unsigned long long *)counts;
    // The table is on the device, so the rule cannot see how even the partitions
    // are, and an edge-balanced cut of a degree-ordered graph puts every isolated
    // vertex into one.  A partition per block therefore only where the widest that
    // the call can have stays cheap: 2,048 words in all, 512 per partition on
    // average (four partitions, one with nearly all: 23 us; the spans 8), and two
    // blocks per SM (600 and more partitions: 10 us for the spans, 12 for blocks).
    if (n_words <= kNaWholeWords && n_words <= 512ull * n_parts && n_parts <= 2 * sms) {
        k_na_whole<<<n_parts, kNaBlock, 0, s>>>(in, cp, cnt, routes);
    } else {
        k_na_zero<<<(3 * n_parts + 255) / 256, 256, 0, s>>>(cnt, 3ull * n_parts);
        // two turns of 4 words per warp at least, up to 8 blocks per SM
        const unsigned long long warps = 8ull * sms * (kNaSpanBlock / 32);
        const unsigned long long span =
            n_words <= kNaSpanWords * warps ? kNaSpanWords : ((n_words + warps - 1) / warps + 3) / 4 * 4;
        const unsigned long long spans = (n_words + span - 1) / span;
        cudaLaunchAttribute early{};
        early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        early.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg{};
        cfg.stream = s;
        cfg.attrs = &early;
        // plain launches in a capture: a graph of the caller's keeps plain edges
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) cudaGetLastError();
        cfg.numAttrs = cap == cudaStreamCaptureStatusNone ? 1 : 0;
        cfg.gridDim = dim3((unsigned int)((spans * 32 + kNaSpanBlock - 1) / kNaSpanBlock));
        cfg.blockDim = dim3(kNaSpanBlock);
        cudaError_t e = cudaLaunchKernelEx(&cfg, k_na_spans, in, span, cnt);
        cfg.gridDim = dim3((n_parts + 255) / 256);
        cfg.blockDim = dim3(256);
        if (e == cudaSuccess)
            e = cudaLaunchKernelEx(&cfg, k_na_select, in, (const unsigned long long *)cnt, cp, (unsigned char *)routes);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return HYTG_ERR_CUDA;
        }
    }
    return cudaGetLastError() == cudaSuccess ? HYTG_OK : HYTG_ERR_CUDA;
}
