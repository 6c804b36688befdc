// Engine selection of Sec. V-A (Eq. 1-3 and the selection rule), shared by
// the planning kernels.  RTT = 1; alpha, beta, gamma are rationals over
// kParamDen, so every comparison is exact in 128-bit integers.
#pragma once

#include "common.cuh"

namespace hytg {

// ceil(x / d); by shifts when d is a power of two, as the paper's m and MR are
// (the decision is on the critical path of every iteration).
__device__ __forceinline__ unsigned long long div_up(unsigned long long x, unsigned long long d) {
    if ((d & (d - 1)) == 0) {
        const int s = __ffsll((long long)d) - 1;
        return (x >> s) + ((x & (d - 1)) != 0);
    }
    const unsigned long long q = x / d;
    return q + (x != q * d);
}

__device__ __forceinline__ int decide_route_counts(unsigned int p, unsigned long long Ei,
                                                   unsigned long long A, unsigned long long Ae,
                                                   unsigned long long L, const CostParams &cp) {
    if (Ae == 0) return kRouteNone;
    const bool resident = p < cp.n_cached;
    if (cp.force_route == kRouteCache && resident) return kRouteCache;
    if (cp.force_route == kRouteF || cp.force_route == kRouteC || cp.force_route == kRouteZ)
        return cp.force_route;
    if (cp.force_route == 5) {
        const unsigned long long h =
            mix64(cp.seed ^ mix64(((unsigned long long)cp.iteration << 32) | p));
        if (resident) return 1 + (int)(h % 4ull);   // cache, F, C, Z
        return 2 + (int)(h % 3ull);                 // F, C, Z
    }
    if (resident) return kRouteCache;
    typedef unsigned __int128 u128;
    // the quotients' operands are byte and line counts of one partition, far
    // below 2^64, so they divide in 64 bits (a 128-bit division is a slow
    // software routine); the products below are taken in 128 bits
    const unsigned long long den = cp.m * cp.MR;
    const u128 Tef = div_up(Ei * cp.d1, den);
    const u128 Tec = div_up(Ae * cp.d1 + A * cp.d2, den);
    const u128 Tl = div_up(L, cp.MR);
    // Tiz = Tl * (gamma + (1 - gamma) * Ae / Ei) = TizN / TizD
    const u128 TizN = Tl * ((u128)cp.gamma_num * Ei + (u128)(kParamDen - cp.gamma_num) * Ae);
    const u128 TizD = (u128)kParamDen * Ei;
    const bool c1 = (u128)kParamDen * Tec < (u128)cp.alpha_num * Tef;
    const bool c2 = (u128)kParamDen * Tec * TizD < (u128)cp.beta_num * TizN;
    if (c1 && c2) return kRouteC;
    if (Tef * TizD < TizN) return kRouteF;
    return kRouteZ;
}

}  // namespace hytg
