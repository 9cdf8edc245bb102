// Packing and unfolding of the pair-adapted ladder, shared by its BF16 (ladder_tc.cu) and FP64
// (pairs64.cu) forms.  Internal linkage: include from kernel files only.
#pragma once

#include "common.cuh"

namespace adc {
namespace {

// ---- pair-adapted ladder: operands and result ---------------------------------------
// A v x v matrix x as its pairs c >= d, p = c (c + 1) / 2 + d: half 0 x_cd + x_dc, half 1
// x_cd - x_dc, each handed to put(half, row, p, value).  Matrix m of the input: element (r, s) at
// in[base(m) + r * rs + s].
//   integrals: m -> a = a0 + m / nb, b = m % nb (b <= a, others skipped), the matrix
//     (ac|bd) over (c, d), row a (a + 1) / 2 + b less put.row0; the diagonal c = d holds 2 (ac|bc)
//   vectors: matrix m is row m; the diagonal holds x_cc
// Bound by HBM: every element is read once (32 x 32 tiles, the mirrored tile through shared
// memory).
template <typename Tin, typename Put>
__global__ void __launch_bounds__(256) k_pair_pack(const Tin* __restrict__ in, int v, long long nmat, long long ms,
                                                   long long rs, int integrals, int a0, int nb, Put put) {
    __shared__ Tin t1[32][33], t2[32][33];
    const int nt = (v + 31) / 32;
    const long long ntri = (long long)nt * (nt + 1) / 2;
    const int tx = threadIdx.x, ty = threadIdx.y;
    for (long long u = blockIdx.x; u < nmat * ntri; u += gridDim.x) {
        const long long m = u / ntri;
        int r = (int)(u - m * ntri), ct = (int)((sqrtf(8.0f * r + 1.0f) - 1.0f) * 0.5f);
        while ((ct + 1) * (ct + 2) / 2 <= r) ++ct;
        while (ct * (ct + 1) / 2 > r) --ct;
        const int dt = r - ct * (ct + 1) / 2, c0 = ct * 32, d0 = dt * 32;
        long long row = m, base = m * ms;
        if (integrals) {
            const long long a = m / nb, b = m - a * nb;
            if (b > a0 + a) continue;  // uniform over the block
            row = (a0 + a) * (a0 + a + 1) / 2 + b - put.row0;
            base = a * v * rs + b * v;
        }
        for (int i = ty; i < 32; i += 8) {
            const int cc = c0 + i, dd = d0 + tx;
            t1[i][tx] = cc < v && dd < v ? in[base + (long long)cc * rs + dd] : (Tin)0;
            const int c2 = d0 + i, d2 = c0 + tx;  // the mirrored tile: rows d, columns c
            t2[i][tx] = c2 < v && d2 < v ? in[base + (long long)c2 * rs + d2] : (Tin)0;
        }
        __syncthreads();
        for (int i = ty; i < 32; i += 8) {
            const int cc = c0 + i, dd = d0 + tx;
            if (cc < v && dd <= cc) {
                const Tin x = t1[i][tx], y = t2[tx][i];
                const long long p = (long long)cc * (cc + 1) / 2 + dd;
                put(0, row, p, dd == cc && !integrals ? x : x + y);
                put(1, row, p, x - y);
            }
        }
        if (ct == nt - 1 && dt == nt - 1 && ty == 0) put.pad(row, tx);
        __syncthreads();
    }
}

// S and A of one pair and matrix, the sums over the K slices, as (S + A) / 2 and (S - A) / 2.
__device__ __forceinline__ void pair_sums(const double* T0, const double* T1, int slices, long long part, double& u, double& w) {
    double S = 0.0, A = 0.0;
    for (int k = 0; k < slices; ++k) {
        S += T0[k * part];
        A += T1[k * part];
    }
    u = 0.5 * (S + A);
    w = 0.5 * (S - A);
}
// FP32 slices: summed as pairs of FP32 numbers (two-sum, 48 bits), since the FP64 pipe's two operations
// per cycle and SM would bound the kernel (745 us for 160 matrices of 400 x 400 with FP64 sums)
__device__ __forceinline__ void two_sum(float& hi, float& lo, float x) {
    const float s = hi + x, b = s - hi;
    lo += (hi - (s - b)) + (x - b);
    hi = s;
}
__device__ __forceinline__ void pair_sums(const float* T0, const float* T1, int slices, long long part, double& u, double& w) {
    float sh = 0.0f, sl = 0.0f, ah = 0.0f, al = 0.0f;
    for (int k = 0; k < slices; ++k) {
        two_sum(sh, sl, T0[k * part]);
        two_sum(ah, al, T1[k * part]);
    }
    float uh = sh, ul = sl + al, wh = sh, wl = sl - al;
    two_sum(uh, ul, ah);
    two_sum(wh, wl, -ah);
    u = (double)(0.5f * uh) + (double)(0.5f * ul);
    w = (double)(0.5f * wh) + (double)(0.5f * wl);
}

// out[m][a][b] += (S + A) / 2 and out[m][b][a] += (S - A) / 2 for the pairs a >= b, with S and A
// the FP64 sums over the K slices of T0[slice][p][m] and T1 (p = a (a + 1) / 2 + b).
// 16 x 16 pair tiles x 8 matrices through shared memory: T is read in whole sectors along m, out
// updated along its rows in both orientations.
template <typename Tt>
__global__ void __launch_bounds__(256) k_pair_unfold(const Tt* __restrict__ T0, const Tt* __restrict__ T1, int slices,
                                                     long long P, int nm, int v, double* __restrict__ out) {
    __shared__ double u[8][16][17], w[8][16][17];
    const int nt = (v + 15) / 16, nmt = (nm + 7) / 8;
    const long long ntri = (long long)nt * (nt + 1) / 2, part = P * nm;
    for (long long blk = blockIdx.x; blk < ntri * nmt; blk += gridDim.x) {
        const int r = (int)(blk / nmt), m0 = (int)(blk % nmt) * 8;
        int at = (int)((sqrtf(8.0f * r + 1.0f) - 1.0f) * 0.5f);
        while ((at + 1) * (at + 2) / 2 <= r) ++at;
        while (at * (at + 1) / 2 > r) --at;
        const int bt = r - at * (at + 1) / 2, a0 = at * 16, b0 = bt * 16;
        const int mi = threadIdx.x & 7, m = m0 + mi;
        for (int e = threadIdx.x >> 3; e < 256; e += 32) {
            const int a = a0 + e / 16, b = b0 + e % 16;
            if (a < v && b <= a && m < nm) {
                const long long t = ((long long)a * (a + 1) / 2 + b) * nm + m;
                pair_sums(T0 + t, T1 + t, slices, part, u[mi][e / 16][e % 16], w[mi][e / 16][e % 16]);
            }
        }
        __syncthreads();
        for (int e = threadIdx.x; e < 8 * 256; e += 256) {
            const int k = e / 256, i = (e / 16) % 16, j = e % 16, mm = m0 + k;
            if (mm >= nm) continue;
            if (a0 + i < v && b0 + j <= a0 + i) out[((long long)mm * v + a0 + i) * v + b0 + j] += u[k][i][j];
            // the mirrored tile: rows b, columns a > b
            if (b0 + i < v && a0 + j < v && b0 + i < a0 + j) out[((long long)mm * v + b0 + i) * v + a0 + j] += w[k][j][i];
        }
        __syncthreads();
    }
}

}  // namespace
}  // namespace adc
