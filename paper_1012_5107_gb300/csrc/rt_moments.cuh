// rt_moments.cuh -- sums of image values and of their products to more than
// FP64's precision on the FP32 pipe (rt_split.cuh's error-free transformations),
// for the moments of the cross-correlation.
#pragma once

#include "rt_split.cuh"

namespace grt {

// Values that the three-float sums take: zero, or a magnitude in [2^-40, 2^48).
// The products' remainders stay clear of underflow, and the products, below
// 2^96, of overflow in any sum of up to 2^31 of them: a column's sum runs over
// the rows of a chunk, which may be the whole image.
__device__ __forceinline__ bool xcorr_plain(float v)
{
    const uint32_t u = __float_as_uint(v) & 0x7fffffffu;
    return u == 0u || u - (87u << 23) < (88u << 23);
}

// Three-float running sums of a pair of values; xcorr_low adds remainders.
__device__ __forceinline__ void xcorr_low(Z3& s, float2 v)
{
    const Z2 t = two_sum(s.m, v);
    s.m = t.h;
    s.l = vadd(s.l, t.l);
}
__device__ __forceinline__ void xcorr_add(Z3& s, float2 v)
{
    const Z2 t = two_sum(s.h, v);
    s.h = t.h;
    xcorr_low(s, t.l);
}

}  // namespace grt
