// Small kernels of the device-driven iteration loop.  The host captures one
// iteration (pre-step, counts, selection with the loop's decision, binning,
// cache and zero-copy relax, and with "device_loop" 2 one IF node per
// partition that copies it into a staging slot and relaxes it, and an IF node
// for the C route) as the body of a CUDA-graph WHILE node; k_select ends the
// loop when the frontier is empty, when the iteration cap is reached, when
// the selection (Sec. V-A) sent a partition to a route the body does not hold
// (F or C with "device_loop" 1; a C route larger than the compaction buffer),
// whose copies the host then issues, or when the host has set the cancel word
// (the run passed its deadline).  Iterations run in the body cost no host
// round trip.
#include "common.cuh"

namespace hytg {

namespace {

__global__ void k_zero_u64(unsigned long long *p, unsigned long long n) {
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x)
        p[i] = 0ull;
}

// F copy inside the device loop without a memcpy node: 16-byte loads from
// mapped host memory, coalesced, into the staging slot.
__global__ void k_copy_words(const unsigned int *src, unsigned int *dst, unsigned long long n,
                             const LoopCtl *loop) {
    if (loop && !loop->work) return;
    const unsigned long long n4 = n / 4;
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    const unsigned long long t0 = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    for (unsigned long long i = t0; i < n4; i += stride)
        ((uint4 *)dst)[i] = __ldcs((const uint4 *)src + i);
    for (unsigned long long i = n4 * 4 + t0; i < n; i += stride) dst[i] = src[i];
}

}  // namespace

cudaError_t launch_zero_u64(unsigned long long *p, unsigned long long n, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    unsigned long long blocks = (n + 255) / 256;
    if (blocks > 4ull * device_sms()) blocks = 4ull * device_sms();
    k_zero_u64<<<(unsigned int)blocks, 256, 0, s>>>(p, n);
    return cudaGetLastError();
}

cudaError_t launch_copy_words(const unsigned int *src, unsigned int *dst, unsigned long long n,
                              const LoopCtl *loop, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    if (((uintptr_t)src | (uintptr_t)dst) & 15) return cudaErrorInvalidValue;
    unsigned long long blocks = (n / 4 + 255) / 256;
    if (blocks > 4ull * device_sms()) blocks = 4ull * device_sms();
    if (blocks == 0) blocks = 1;
    k_copy_words<<<(unsigned int)blocks, 256, 0, s>>>(src, dst, n, loop);
    return cudaGetLastError();
}

}  // namespace hytg
