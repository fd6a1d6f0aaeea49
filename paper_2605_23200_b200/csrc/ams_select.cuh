// Device helpers of the mass kernel of libams: the Eq. 1 weight and the fixed-point images of the mass.  Not used by
// the CPU oracle.
#pragma once
#include <float.h>

#include "ams_common.cuh"

namespace ams {
namespace sel {

__device__ __forceinline__ float weight_of(float u, float eps)
{
    // Eq. 1 numerator: max(u, 0) + eps; NaN counts as 0, +inf as FLT_MAX.
    return fminf(__fadd_rn(fmaxf(u, 0.0f), eps), FLT_MAX); // (the sum is never NaN: fmaxf drops a NaN operand)
}

// ---- fixed-point images through fp32 / fp64 arithmetic ------------------------------------------
// Exponent e = ilogb(mx) + 1 of the largest weight mx > 0 (any fp32, subnormals included).
__device__ __forceinline__ int fix_exponent(float mx)
{
    const long long bits = __double_as_longlong((double)mx);
    return (int)((bits >> 52) & 0x7ff) - 1023 + 1;
}

// The fixed-point image A = floor(x * 2^(kFixBits - e)) (0 <= x < 2^e) equals trunc(x) * 2^(kFixBits - e), where
// trunc(x) is x with the mantissa bits below the image's last bit cleared: x = m * 2^(E - 23), and the image
// drops the lowest n = e - 13 - E bits of m when that is positive (all 24 of them from n = 24 on).  So the
// image is available as a double with one conversion and one exact multiplication by a power of two, and
// sums of images (integers below 2^53) can be added in fp64 in any order.
// The truncation takes two additions: below c = 2^(e - 13) a float is cut to a multiple of the image's
// last bit 2^(e - 36) by adding c rounded down (sums in [c, 2c) have exactly that spacing) and taking c off
// again (exact); from c upwards every float is such a multiple already.  c may be subnormal or zero for
// tiny e: then every float is a multiple of the last bit and both branches return x.
__device__ __forceinline__ float fixed_trunc_by_add(float x, float c)
{
    return x >= c ? x : __fsub_rn(__fadd_rd(x, c), c);
}
__device__ __forceinline__ float fixed_trunc_threshold(int e)
{
    const int k = e - (kFixBits - 23); // 2^k, any k in [-161, 115]
    return k >= -126 ? __uint_as_float((unsigned)(k + 127) << 23) : (k >= -149 ? __uint_as_float(1u << (k + 149)) : 0.0f);
}

// 2^(kFixBits - e) as a double (e = fix_exponent of a positive fp32, so the result is a normal double).
__device__ __forceinline__ double fix_scale_of(int e)
{
    return __longlong_as_double((long long)(1023 + kFixBits - e) << 52);
}

// floor(y) for 0 <= y < 2^51 as an integer: y + 2^52 rounded down lands on the integer grid.
__device__ __forceinline__ u64 floor_to_u64(double y)
{
    return (u64)__double_as_longlong(__dadd_rd(y, 4503599627370496.0)) & 0xfffffffffffffull;
}

} // namespace sel
} // namespace ams
