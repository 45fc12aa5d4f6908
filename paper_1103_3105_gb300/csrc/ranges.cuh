// ranges.cuh -- which of a sorted array's groups (equal keys) a CTA runs: those
// that begin in its slice of positions, to the end of the last of them.
#pragma once
#include "common.cuh"

namespace gtx {

// first position in [lo, hi) whose key is not `key` (hi if none; keys sorted);
// the whole CTA (T threads) calls it
template <int T>
__device__ __forceinline__ uint32_t first_other(const uint32_t *keys, uint32_t lo, uint32_t hi, uint32_t key, uint32_t *s_min)
{
    const uint32_t tid = threadIdx.x;
    uint32_t span = T;                // the next T positions, then T probes a round
    while (lo < hi) {
        const uint32_t len = hi - lo;
        const uint32_t step = span == 0 ? (len + T - 1) / T : 1;
        if (tid == 0) *s_min = T;
        __syncthreads();
        const uint64_t at = (uint64_t)lo + (uint64_t)(tid + 1) * step - 1;
        const uint32_t p = at < hi ? (uint32_t)at : hi - 1;
        const uint32_t m = __ballot_sync(kFull, __ldg(&keys[p]) != key);
        if ((tid & 31) == 0 && m) atomicMin(s_min, tid + (uint32_t)__ffs(m) - 1);
        __syncthreads();
        const uint32_t i = *s_min;
        __syncthreads();
        if (i == T) {                 // none among the probes, the last of which was min(...) below
            if (step > 1 || len <= (uint32_t)T) return hi;
            lo += T;
        } else {
            const uint32_t a = lo + i * step;
            if (step == 1) return a < hi ? a : hi - 1;
            hi = a + step < hi ? a + step : hi;
            lo = a;
        }
        span = 0;
    }
    return hi;
}

// the range of this CTA (blockIdx.x-th slice of n positions): from the first
// head at or after the slice's start to the first at or after its end; false if
// no group begins in it.  The whole CTA (T threads) calls it.
template <int T>
__device__ __forceinline__ bool group_range(const uint32_t *keys, uint32_t n, uint32_t slice, uint32_t *s_min,
                                            uint32_t &lo, uint32_t &hi)
{
    const uint64_t s0_ = (uint64_t)blockIdx.x * slice;
    lo = 0;
    hi = n;
    if (s0_ >= n) return false;
    const uint32_t s0 = (uint32_t)s0_;
    const uint32_t s1 = n - s0 < slice ? n : s0 + slice;
    if (s0 > 0) {
        const uint32_t k = __ldg(&keys[s0 - 1]);
        if (__ldg(&keys[s1 - 1]) == k) return false;   // the slice lies inside an earlier slice's group
        lo = first_other<T>(keys, s0, s1, k, s_min);
    }
    if (s1 < n) hi = first_other<T>(keys, s1, n, __ldg(&keys[s1 - 1]), s_min);
    return true;
}

}  // namespace gtx
