// Reductions within a warp.
#pragma once

namespace adc {

// Sums N (a power of two, <= 32) values per lane over the warp: each step exchanges half of the values
// that are left, N - 1 additions per lane instead of 5 N (the FP64 units' two a cycle per SM bound the
// reduction of a 8 x 4 block of inner products: 20 -> 14 us a call at some 30 x 4 vectors of 16,245, of
// which the products' own FP64 is 9).  v[0] of lane l is value l N / 32.
template <int N>
__device__ __forceinline__ void warp_fold(double (&v)[N], int lane) {
    int off = 16;
#pragma unroll
    for (int m = N; m > 1; m >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int i = 0; i < m / 2; ++i) {
            const double give = up ? v[i] : v[i + m / 2], keep = up ? v[i + m / 2] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, off);
        }
        off >>= 1;
    }
#pragma unroll
    for (int s = 32 / N; s > 1; s >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], s / 2);
}

}  // namespace adc
