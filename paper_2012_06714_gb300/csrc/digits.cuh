// The integer arithmetic of gemm64.cu: a double as digits, and sums of digit products as a double.
#pragma once

#include <cstdint>
#include <cstring>

#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace adc {

constexpr int ND = 8;         // digits
constexpr int SMIN = ND - 1;  // lowest weight kept
constexpr int NL = 8;         // weights SMIN .. 2 (ND - 1)

// The exponent field of a double as the rows' scales count it: subnormal numbers have that of the smallest
// normal ones.
__host__ __device__ __forceinline__ int exponent_of(uint64_t b) {
    const int e = (int)(b >> 52) & 0x7ff;
    return e > 0 ? e : 1;
}

// x (its bits) in a row of largest exponent field ef -> round(x 2^(1085 - ef)), below 2^63 in size (the row's
// scale is 2^(ef - 1022)); 0 in a row that is not finite.  Integer arithmetic only: the FP64 pipe (2 operations
// per cycle and SM) would be the bound.
__host__ __device__ __forceinline__ long long scaled_integer(uint64_t b, int ef) {
    const int sh = ef - exponent_of(b) - 10;  // right shift of the 53-bit significand (-10: ten more bits)
    if (ef >= 0x7ff || sh >= 55) return 0;
    const long long m = (long long)(b & 0xfffffffffffffULL) | ((b << 1) >> 53 ? 1LL << 52 : 0);
    const long long v = sh <= 0 ? m << -sh : (m + (1LL << (sh - 1))) >> sh;
    return (long long)b < 0 ? -v : v;
}

// Digit p < 7 of v is the p-th byte of v + sum_p 128 256^p less 128: the carries in one addition; the top one
// is in [-128, 128].
__host__ __device__ __forceinline__ uint64_t with_carries(long long v) { return (uint64_t)v + 0x0080808080808080ULL; }
__host__ __device__ __forceinline__ int digit(long long v, uint64_t w, int p) {
    if (p < ND - 1) return (int)((w >> (8 * p)) & 0xff) - 128;
    return v >= 0 ? (int)(w >> 56) : (int)((long long)w >> 56);
}

__host__ __device__ __forceinline__ int leading_zeros(uint64_t x) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)x);
#else
    return __builtin_clzll(x);
#endif
}

// (hi 2^32 + lo) 2^e, rounded to nearest, by integer arithmetic; |hi| < 2^62
__host__ __device__ __forceinline__ double to_double(long long hi, long long lo, int e) {
    long long H = hi + (lo >> 32);
    uint32_t L = (uint32_t)lo;
    const bool neg = H < 0;
    if (neg) {
        L = 0u - L;
        H = L == 0 ? -H : ~H;
    }
    uint64_t m;
    int top;  // weight of m's bit 63
    if (H != 0) {
        const int lz = leading_zeros((uint64_t)H);
        const uint64_t l = (uint64_t)L << 32;
        m = ((uint64_t)H << lz) | (lz ? l >> (64 - lz) : 0ull);
        top = 95 - lz;
    } else {
        if (L == 0) return 0.0;
        const int lz = leading_zeros((uint64_t)L) - 32;
        m = (uint64_t)L << (32 + lz);
        top = 31 - lz;
    }
    m = (m >> 11) + ((m >> 10) & 1);  // 53 bits, carry into bit 53 raises the exponent below
    const int be = top + e + 1023;
    uint64_t bits;
    if (be > 2046)
        bits = 0x7ffull << 52;
    else if (be > 0)
        bits = m + ((uint64_t)(be - 1) << 52);
    else  // below the normal range (rounded once more)
        bits = be < -52 ? 0 : (m >> (1 - be)) + ((m >> -be) & 1);
    bits |= neg ? 1ull << 63 : 0ull;
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)bits);
#else
    double x;
    std::memcpy(&x, &bits, sizeof x);
    return x;
#endif
}

}  // namespace adc
