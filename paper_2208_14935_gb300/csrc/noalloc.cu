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

constexpr unsigned int kNaBlock = 256;

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

__device__ __forceinline__ int na_route(const NaInput &in, unsigned int p, unsigned long long act,
                                        unsigned long long edges, unsigned long long lines, const CostParams &cp) {
    return decide_route_counts(p, in.off[na_bound(in, p + 1)] - in.off[na_bound(in, p)], act, edges, lines, cp);
}

// |A_i|, active edges and 128-byte lines (footnote to Eq. 3) of one slice of
// one partition per block: block p * slices + x takes every slices-th group of
// 32 words of partition p.  A warp takes four consecutive words at a time and
// has their offsets in flight together.  One slice: the block holds the whole
// partition, so it also selects the route and one launch does everything;
// several slices add into counts (zeroed before), and k_na_select follows.
//
// What bounds a small call is launches and the chain of dependent loads.  A
// bounds pass, counts with three atomics per word on a few dozen partitions
// and a selection pass took 42 us on 65,536 vertices in 72 partitions; now
// 8.4 us a call, most of it the launch and its caller.
template <bool WHOLE>
__global__ void __launch_bounds__(kNaBlock) k_na_count(NaInput in, unsigned int slices, CostParams cp,
                                                       unsigned long long *counts, unsigned char *routes) {
    __shared__ unsigned long long s_sum[kNaBlock / 32][3];
    const unsigned int p = WHOLE ? blockIdx.x : blockIdx.x / slices, x = WHOLE ? 0 : blockIdx.x % slices;
    const unsigned int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned long long n_words = (in.V + 31) / 32;
    // a word belongs to the last partition that starts at or before it
    const unsigned long long w_lo = p == 0 ? 0 : (na_bound(in, p) + 31) / 32;
    const unsigned long long w_hi = p + 1 == in.n_parts ? n_words : (na_bound(in, p + 1) + 31) / 32;
    unsigned long long act = 0, edges = 0, lines = 0;
    const unsigned long long step = (unsigned long long)slices * (kNaBlock / 32) * 4;
    for (unsigned long long w0 = w_lo + ((unsigned long long)x * (kNaBlock / 32) + wid) * 4; w0 < w_hi; w0 += step) {
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
            act += (bits[q] >> lane) & 1u;
            if (o1[q] > o0[q]) {
                edges += o1[q] - o0[q];
                lines += in.n_arrays *
                         (in.m_shift >= 0 ? ((o1[q] * 4ull - 1) >> in.m_shift) - ((o0[q] * 4ull) >> in.m_shift) + 1
                                          : lines_spanned(o0[q] * 4ull, (o1[q] - o0[q]) * 4ull, in.m));
            }
        }
    }
    act = warp_sum_u64(act);
    edges = warp_sum_u64(edges);
    lines = warp_sum_u64(lines);
    if (lane == 0) {
        s_sum[wid][0] = act;
        s_sum[wid][1] = edges;
        s_sum[wid][2] = lines;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        unsigned long long t = 0;
#pragma unroll
        for (unsigned int w = 0; w < kNaBlock / 32; ++w) t += s_sum[w][threadIdx.x];
        if (WHOLE) {
            counts[3ull * p + threadIdx.x] = t;
            s_sum[0][threadIdx.x] = t;
        } else if (t) {
            atomicAdd(&counts[3ull * p + threadIdx.x], t);
        }
    }
    if (WHOLE) {
        __syncwarp();
        if (threadIdx.x == 0)
            routes[p] = (unsigned char)na_route(in, p, s_sum[0][0], s_sum[0][1], s_sum[0][2], cp);
    }
}

__global__ void k_na_select(NaInput in, const unsigned long long *counts, CostParams cp, unsigned char *routes) {
    const unsigned int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < in.n_parts)
        routes[p] = (unsigned char)na_route(in, p, counts[3ull * p], counts[3ull * p + 1], counts[3ull * p + 2], cp);
}

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
    // One block per partition while a partition's words are few (up to 64 on
    // average; a warp takes 32 per turn of its block, and skewed graphs have
    // partitions of many times the average) or the partitions alone fill the
    // chip; else slices of 32 words or more, up to 8 blocks per SM in all, at
    // the price of a memset and a second kernel.  Measured per call: 28 words
    // on average 8.4 us whole; 128 words on a skewed graph (909,625 vertices,
    // 222 partitions) 26 us whole, 18 us sliced.
    const unsigned long long words = (V + 31) / 32 / n_parts;
    unsigned long long slices = 1;
    if (words > 64) {
        slices = 8ull * sms / n_parts;
        if (slices > words / 32) slices = words / 32;
        if (slices < 1) slices = 1;
    }
    unsigned long long *cnt = (unsigned long long *)counts;
    if (slices == 1) {
        k_na_count<true><<<n_parts, kNaBlock, 0, s>>>(in, 1, cp, cnt, routes);
    } else {
        if (cudaMemsetAsync(cnt, 0, 24ull * n_parts, s) != cudaSuccess) {
            cudaGetLastError();
            return HYTG_ERR_CUDA;
        }
        k_na_count<false><<<(unsigned int)(n_parts * slices), kNaBlock, 0, s>>>(in, (unsigned int)slices, cp, cnt, routes);
        k_na_select<<<(n_parts + 255) / 256, 256, 0, s>>>(in, cnt, cp, routes);
    }
    return cudaGetLastError() == cudaSuccess ? HYTG_OK : HYTG_ERR_CUDA;
}
