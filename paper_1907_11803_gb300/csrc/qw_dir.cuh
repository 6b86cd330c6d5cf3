// qw_dir.cuh -- integer helpers of the bucket-range search (virtual
// rehashing, Section 2), shared by the query kernels.
#pragma once

#include <stdint.h>

namespace qw {

// floor(a / R) for R > 0 (C division truncates toward zero): for a < 0 it is
// ~(~a / R).  Bucket ids and radii nearly always fit 32 bits, where the division
// is a fraction of the 64-bit one's instructions.
__device__ __forceinline__ int64_t floordiv64(int64_t a, int64_t R)
{
    const int64_t sign = a >> 63;
    const uint64_t u = (uint64_t)(a ^ sign), r = (uint64_t)R;
    const uint64_t q = ((u | r) >> 32) ? u / r : (uint64_t)((uint32_t)u / (uint32_t)r);
    return (int64_t)q ^ sign;
}

__device__ __forceinline__ int64_t clamp64(int64_t x, int64_t lo, int64_t hi)
{
    return x < lo ? lo : (x > hi ? hi : x);
}

// Offset (inside the tile's entry segment) of the first entry with bid >= x.
// The directory of a tile holds its distinct bids ub[0..cnt) ascending and the
// offset uo[] of each bid's first entry.  When every bid between ub[0] and x is
// present the answer sits at slot x - ub[0]; otherwise binary search.
__device__ __forceinline__ int dir_lower(const int32_t *__restrict__ ub,
                                         const int32_t *__restrict__ uo, int cnt, int len,
                                         int64_t x)
{
    if (cnt == 0) return 0;
    const int32_t b0 = ub[0];
    if (x <= b0) return 0;
    const int64_t p = x - b0;
    if (p < cnt && ub[p] == x) return uo[p];
    int lo = 0, hi = cnt;
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if ((int64_t)ub[mid] < x) lo = mid + 1; else hi = mid;
    }
    return lo < cnt ? uo[lo] : len;
}

}  // namespace qw
