// Conversions between FP64 and the float-float pair hi = fl32(x), lo = fl32(x - hi) on the integer pipe.
// The state copies convert every value; as FP64 instructions (2 lanes a clock and SM) the four of a split
// and the three of a join bounded them (mixed P3, 1,572,864 elements: 1.1 ms where the memory needs
// 0.4 ms).  The results are those of the FP64 instructions for every input: values outside the range
// handled with integers take those instructions.
#pragma once

#include <cstdint>

namespace dg {
namespace ff {

// x as a double, exactly
__device__ __forceinline__ double widen(float x) {
    const uint32_t b = __float_as_uint(x), e = b & 0x7f800000u;
    if (e == 0u || e == 0x7f800000u) return (b << 1) == 0u ? __hiloint2double((int)b, 0) : (double)x;
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}

// |x| with 2^-74 <= |x| < 2^126: neither part leaves FP32's normal range, except lo = 0
__device__ __forceinline__ bool in_range(uint64_t b) {
    const uint32_t e = (uint32_t)(b >> 52) & 0x7ffu;
    return e - (1023u - 74u) < 200u;
}

// hi = fl32(x): the 29 low bits of the mantissa rounded to nearest, ties to even
__device__ __forceinline__ uint32_t round_bits(uint64_t b) {
    const uint64_t r = b + 0x0fffffffull + ((b >> 29) & 1ull);
    return ((uint32_t)(b >> 32) & 0x80000000u) | (((uint32_t)(r >> 29) - 0x40000000u * 7u) & 0x7fffffffu);
}

__device__ __forceinline__ float narrow(double x) {
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    if (!in_range(b)) return (b << 1) == 0ull ? __uint_as_float((uint32_t)(b >> 32)) : (float)x;
    return __uint_as_float(round_bits(b));
}

__device__ __forceinline__ void split(double x, float& hi, float& lo) {
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    if (!in_range(b)) {
        if ((b << 1) == 0ull) {   // x - hi = +0
            hi = __uint_as_float((uint32_t)(b >> 32));
            lo = 0.f;
        } else {
            hi = (float)x;
            lo = (float)(x - (double)hi);
        }
        return;
    }
    const uint64_t r = b + 0x0fffffffull + ((b >> 29) & 1ull);
    hi = __uint_as_float(round_bits(b));
    // x - hi in units of 2^(E - 52): the low bits, less one unit of hi if it was rounded up
    int32_t d = (int32_t)((uint32_t)b & 0x1fffffffu);
    if (((r ^ b) >> 29) & 1ull) d -= 1 << 29;   // the last kept bit changed: rounded up
    if ((int64_t)b < 0) d = -d;
    const uint32_t e = (uint32_t)(b >> 52) & 0x7ffu;   // scale 2^(e - 1023 - 52)
    lo = (float)d * __uint_as_float((e - 1023u - 52u + 127u) << 23);
}

__device__ __forceinline__ double join(float hi, float lo) { return widen(hi) + widen(lo); }

}  // namespace ff
}  // namespace dg
