// pf_ancestor.cuh -- shared pieces of the ancestor kernels (Gumbel-max, Metropolis, rejection).
#pragma once
#include "pf_device.cuh"
#include "pf_internal.h"

namespace pfk {

// The tracker g of CTA b: cta_prefix[g] <= b < cta_prefix[g + 1] (bisection; every tracker
// has at least one CTA, so the prefix is strictly increasing).
__device__ __forceinline__ int ancestor_tracker(const AncestorLaunch &G, int b) {
    int lo = 0, hi = G.ntrk - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(G.cta_prefix + mid) <= b) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Rejection: offspring per CTA of a tracker of n particles (a multiple of 32).  Small trackers are
// spread over the SMs (kRejectionSpread CTAs, four on each of the part's 152, while a CTA keeps 32
// offspring): F32 1000 particles in one CTA of at most kRejectionOffspring 77 us a frame, so 14.
// The host numbers the CTAs by the same function, so it depends on n alone.
constexpr int kRejectionSpread = 608;
__host__ __device__ inline int rejection_pool(int64_t n) {
    const int64_t p = ((n + kRejectionSpread - 1) / kRejectionSpread + 31) / 32 * 32;
    return p > kRejectionOffspring ? kRejectionOffspring : static_cast<int>(p);
}

__device__ __forceinline__ double log_uniform(uint32_t w, double) { return log(uniform_f64(w)); }
__device__ __forceinline__ float log_uniform(uint32_t w, float) { return logf(uniform_f32(w)); }

// ln u <= d, u the uniform of word w, exactly as log_uniform(w, A{}) <= d decides it.  In FP64 the
// FP32 hardware logarithm (within 6e-6 of ln u over [2^-24, 1): 3 ulp, and 2^-21.4 above 1/2)
// decides unless the two sides lie within 1e-4 of each other, which one test in thousands
// needs the FP64 logarithm for (about 30 operations at 1.7 a clock and SM): REF64 Metropolis
// at 50003 particles 334 -> 108 us a frame, rejection at 20003 686 -> 155.  (d rounded to FP32
// moves by less than 2e-6 where |d| <= 17; beyond, ln u >= -16.64 is 1e-4 and more away.  NaN
// takes the accurate test and refuses.)  In FP32 the accurate logarithm stays: the kernels wait
// on their gathers, and the shorter test takes registers that residency needs more (rejection
// F16 at 200003 particles 126 against 123 us a frame).
template <typename A>
__device__ __forceinline__ bool log_uniform_le(uint32_t w, A d) {
    if constexpr (sizeof(A) == 8) {
        const float gap = static_cast<float>(d) - __logf(uniform_f32(w));
        if (gap > 1e-4f) return true;
        if (gap < -1e-4f) return false;
    }
    return log_uniform(w, A{}) <= d;
}

}  // namespace pfk
