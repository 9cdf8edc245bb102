// A double as two FP32 numbers, for splits into BF16 planes.
#pragma once

#include <cstdint>
#include <cstring>

#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace adc {

__host__ __device__ __forceinline__ float float_of_bits(uint32_t u) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float f;
    std::memcpy(&f, &u, sizeof f);
    return f;
#endif
}

// x = hi + lo: hi the leading 24 bits of x, lo the other 29 rounded to FP32, so that BF16 planes cut from hi
// and from the remainder plus lo are those of x itself and not of x rounded to FP32.  Integer arithmetic and
// one conversion from an integer: remainders in FP64 (two operations per cycle and SM on this chip) made the
// splits several times slower than their traffic.  lo is exact down to |x| = 2^-74 (below, and above 2^127,
// in FP64; subnormal doubles are 0, as their BF16 planes are).
__host__ __device__ __forceinline__ void two_floats(double x, float& hi, float& lo) {
    uint64_t b;
#ifdef __CUDA_ARCH__
    b = (uint64_t)__double_as_longlong(x);
#else
    std::memcpy(&b, &x, sizeof b);
#endif
    const uint32_t top = (uint32_t)(b >> 32), low = (uint32_t)b, sign = top & 0x80000000u, e = (top >> 20) & 0x7ffu;
    if (e - 949u <= 1149u - 949u) {
        hi = float_of_bits(sign | (e - 896u) << 23 | (top & 0xfffffu) << 3 | low >> 29);
        lo = (float)(int32_t)(low & 0x1fffffffu) * float_of_bits(sign | (e - 948u) << 23);
    } else if (e == 0) {
        hi = float_of_bits(sign);
        lo = 0.0f;
    } else {
        hi = (float)x;
        const double r = x - (double)hi;
        lo = r - r == 0.0 ? (float)r : 0.0f;  // (0 where x or hi is not finite)
    }
}
__host__ __device__ __forceinline__ void two_floats(float x, float& hi, float& lo) {
    hi = x;
    lo = 0.0f;
}

// hi with its last bit set where something follows it: rounded to a BF16 it gives the BF16 nearest to hi + lo
__host__ __device__ __forceinline__ float odd(float hi, float lo) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(__float_as_uint(hi) | (lo != 0.0f ? 1u : 0u));
#else
    uint32_t u;
    std::memcpy(&u, &hi, sizeof u);
    return float_of_bits(u | (lo != 0.0f ? 1u : 0u));
#endif
}

// r + x where |x| is at most |r| or r is 0: the rounded sum, and in x what it leaves out
__host__ __device__ __forceinline__ float add_keep(float r, float& x) {
    const float s = r + x;
    x -= s - r;
    return s;
}

}  // namespace adc
