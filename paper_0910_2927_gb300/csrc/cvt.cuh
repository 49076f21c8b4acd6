// FP32 <-> FP64 conversions on the integer units.  GB300 runs the conversion instructions, like all
// FP64 work, at 1/64 of the FP32 rate, so that kernels which only move data between the two types
// were bound by them and not by memory (splitting 3.1 M complex128 into float-float pairs: 47 us,
// 100 MB).  Normal numbers are re-biased as bit patterns; zeros, subnormals, infinities and NaN
// take the conversion instruction.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace sgn {

// (double)f, exactly.
__device__ __forceinline__ double f2d(float f) {
    const uint32_t b = __float_as_uint(f), e = (b >> 23) & 255u;
    if (e - 1u < 254u)
        return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), (int)(b << 29));
    return (double)f;
}

// (float)d, round to nearest even.
__device__ __forceinline__ float d2f(double d) {
    const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
    const uint32_t e = (hi >> 20) & 2047u;
    if (e - 897u < 253u) {  // the result is normal, also when it rounds up
        // bits 29.. of the 52-bit mantissa stay: 20 of hi, 3 of lo; the other 29 round
        const uint32_t m = (((hi & 0x7fffffffu) - (896u << 20)) << 3) | (lo >> 29);
        const uint32_t rest = lo << 3, half = 0x80000000u;
        const uint32_t up = rest > half || (rest == half && (m & 1u)) ? 1u : 0u;
        return __uint_as_float((hi & 0x80000000u) | (m + up));
    }
    return (float)d;
}

// d as a sum of two floats: hi the nearest one (a tie goes away from zero), lo = (float)(d - hi).
__device__ __forceinline__ float2 d2ff(double d) {
    const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
    const uint32_t e = (hi >> 20) & 2047u;
    if (e - 960u < 189u) {  // 2^-63 <= |d| < 2^126: hi is normal, lo normal or zero
        const uint32_t s = hi & 0x80000000u;
        // the leading 24 bits, rounded by the next one, and the other 29 less that rounding as an
        // integer of at most 28 bits and a sign, times 2^(exponent - 52)
        const int r = (int)(lo << 3) >> 3;
        const uint32_t t = ((((hi & 0x7fffffffu) - (896u << 20)) << 3) | (lo >> 29)) + (r < 0 ? 1u : 0u);
        return make_float2(__uint_as_float(s | t), __int2float_rn(r) * __uint_as_float(s | ((e - 948u) << 23)));
    }
    const float h = (float)d;
    return make_float2(h, (float)(d - (double)h));
}

}  // namespace sgn
