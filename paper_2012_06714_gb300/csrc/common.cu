// Elementwise kernels and the tensor-contraction executor used by setup and
// the FP64 sigma path.
#include <algorithm>
#include <cstring>
#include <map>

#include <cuda_bf16.h>

#include "common.cuh"
#include "split.cuh"
#include "warp.cuh"
#include "gemm64.cuh"
#include "ladder_tc.cuh"

namespace adc {

namespace {

struct PermArgs {
    int nd;
    long long dout[kMaxDim];
    long long sin[kMaxDim];  // input stride for each output axis
};

// the inputs of the permutes: an array, or the FP64 sum of S arrays `stride` apart
template <typename Tin>
struct Plain {
    const Tin* p;
    __device__ Tin operator()(long long i) const { return p[i]; }
};
template <typename Tin>
struct SumOf {
    const Tin* p;
    int S;
    long long stride;
    __device__ double operator()(long long i) const {
        double x = (double)p[i];
        for (int s = 1; s < S; ++s) x += (double)p[s * stride + i];
        return x;
    }
};

// I: the index type of the coordinate arithmetic (32-bit when every offset fits: integer
// division by a runtime divisor is several times cheaper than in 64 bits)
template <typename I, typename In, typename Tout>
__global__ void permute_kernel(In in, Tout* __restrict__ out, PermArgs a, long long total, double alpha, double beta) {
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        I r = (I)idx, off = 0;
        for (int j = a.nd - 1; j >= 0; --j) {
            const I d = (I)a.dout[j];
            const I q = r / d;
            off += (r - q * d) * (I)a.sin[j];
            r = q;
        }
        const double v = alpha * (double)in(off);
        out[idx] = (Tout)((beta == 0.0) ? v : v + beta * (double)out[idx]);
    }
}

__global__ void axpby_kernel(long long n, double alpha, const double* __restrict__ x, double beta, double* __restrict__ y) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = (beta == 0.0) ? alpha * x[i] : alpha * x[i] + beta * y[i];
}

__global__ void fill_kernel(long long n, double v, double* __restrict__ y) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = v;
}

// x as BF16 planes: o0 + o1 (+ o2 where there is a third), each the rounded remainder of those before
template <typename X>
__device__ __forceinline__ void put_planes(X x, long long ad, __nv_bfloat16* o0, __nv_bfloat16* o1, __nv_bfloat16* o2) {
    float f, lo;
    two_floats(x, f, lo);
    const __nv_bfloat16 h = __float2bfloat16(odd(f, lo));
    o0[ad] = h;
    f = add_keep(f - __bfloat162float(h), lo);
    const __nv_bfloat16 m = __float2bfloat16(f);
    o1[ad] = m;
    if (o2) o2[ad] = __float2bfloat16((f - __bfloat162float(m)) + lo);
}

// out[p][r*Kp + k] (two or three BF16 planes) from the permuted input, zero for k >= K
template <typename I, typename Tin>
__global__ void permute_split_kernel(const Tin* __restrict__ in, __nv_bfloat16* __restrict__ o0,
                                     __nv_bfloat16* __restrict__ o1, __nv_bfloat16* __restrict__ o2, PermArgs a,
                                     long long rows, long long K, long long Kp) {
    const long long total = rows * Kp;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const I r = (I)(idx / Kp), k = (I)(idx - (long long)r * Kp);
        Tin x = 0;
        if (k < (I)K) {
            I lin = r * (I)K + k, off = 0;
            for (int j = a.nd - 1; j >= 0; --j) {
                const I d = (I)a.dout[j];
                const I q = lin / d;
                off += (lin - q * d) * (I)a.sin[j];
                lin = q;
            }
            x = in[off];
        }
        put_planes(x, idx, o0, o1, o2);
    }
}

// ---- transposing permutes through shared memory ----------------------------------
// When the output's fastest axis x is strided in the input, the plain kernels above read one
// element per memory sector.  These take a 32 x 32 tile over x and the axis y that is
// contiguous in the input: threads read along y (coalesced), the tile is transposed in shared
// memory, threads write along x (coalesced).  The remaining output axes index the tiles.
struct TileArgs {
    int nrest;
    long long rdim[kMaxDim], rsin[kMaxDim], rsout[kMaxDim];  // other output axes: extent, input / output stride
    long long nx, ny, sx_in, sy_out;  // x: output-innermost axis (input stride sx_in); y: input-contiguous axis
    long long ntx, nty, nblocks;
};

// output of split BF16 planes [rows][Kp] (the linear output index counts [rows][K])
struct OpPlanes {
    __nv_bfloat16 *o0, *o1, *o2;
    long long K, Kp;
    __device__ long long addr(long long lin) const {
        const long long r = lin / K;
        return r * Kp + (lin - r * K);
    }
    template <typename V>
    __device__ void put(long long ad, V x) const {
        put_planes(x, ad, o0, o1, o2);
    }
    template <int V, typename X>
    __device__ void put_n(long long ad, const X (&x)[V]) const {
        if constexpr (V == 4) {
            uint2 w[3];
            float f[4], lo[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) two_floats(x[i], f[i], lo[i]);
#pragma unroll
            for (int p = 0; p < 3; ++p) {
                const __nv_bfloat162 l = p ? __floats2bfloat162_rn(f[0], f[1]) : __floats2bfloat162_rn(odd(f[0], lo[0]), odd(f[1], lo[1])),
                                     h = p ? __floats2bfloat162_rn(f[2], f[3]) : __floats2bfloat162_rn(odd(f[2], lo[2]), odd(f[3], lo[3]));
                w[p] = make_uint2(*(const unsigned*)&l, *(const unsigned*)&h);
                f[0] -= __uint_as_float(w[p].x << 16);
                f[1] -= __uint_as_float(w[p].x & 0xffff0000u);
                f[2] -= __uint_as_float(w[p].y << 16);
                f[3] -= __uint_as_float(w[p].y & 0xffff0000u);
#pragma unroll
                for (int i = 0; i < 4; ++i) f[i] = add_keep(f[i], lo[i]);
            }
            *(uint2*)(o0 + ad) = w[0];
            *(uint2*)(o1 + ad) = w[1];
            if (o2) *(uint2*)(o2 + ad) = w[2];
        } else {
#pragma unroll
            for (int e = 0; e < V; ++e) put(ad + e, x[e]);
        }
    }
    // after the line of `len` elements from lin (at address ad): the row's padding, if it ends there
    __device__ void finish(long long lin, long long len, long long ad, int i, int step) const {
        if (Kp == K || (lin + len) % K) return;
        for (long long k = i; k < Kp - K; k += step) put_planes(0.0f, ad + len + k, o0, o1, o2);
    }
};
// out = alpha x + beta out
template <typename Tout>
struct OpAxpby {
    Tout* out;
    double alpha, beta;
    __device__ long long addr(long long lin) const { return lin; }
    template <typename V>
    __device__ void put(long long ad, V x) const {
        if (alpha == 1.0 && beta == 0.0) {
            out[ad] = (Tout)x;
            return;
        }
        if constexpr (sizeof(V) == 4 && sizeof(Tout) == 4) {
            // +- x (+ out) rounded once, as in FP64 but without its pipe
            if ((alpha == 1.0 || alpha == -1.0) && (beta == 0.0 || beta == 1.0)) {
                const float f = alpha == 1.0 ? x : -x;
                out[ad] = beta == 0.0 ? f : out[ad] + f;
                return;
            }
        }
        const double v = alpha == 1.0 ? (double)x : alpha * (double)x;
        out[ad] = (Tout)(beta == 0.0 ? v : beta == 1.0 ? v + (double)out[ad] : v + beta * (double)out[ad]);
    }
    template <int V, typename X>
    __device__ void put_n(long long ad, const X (&x)[V]) const {
#pragma unroll
        for (int e = 0; e < V; ++e) put(ad + e, x[e]);
    }
    __device__ void finish(long long, long long, long long, int, int) const {}
};

// ---- permutes along lines -----------------------------------------------------------
// When the output's fastest axis is contiguous in the input too, a group of tpl threads copies a
// whole line of it: one coordinate computation per line instead of one per element (the element-wise
// kernels spend most of their time on integer divisions), four loads in flight per thread.
struct LineArgs {
    int nd;  // axes above the line
    long long dout[kMaxDim], sin[kMaxDim];
    long long len, nlines, seg;  // lines are cut into segments of seg elements (a multiple of 4)
    int nseg, tpl;               // segments per line, threads per segment
};
// V elements per thread at a time (4 when the lines' lengths are multiples of it: 8-byte stores of the
// BF16 planes, which 2-byte ones would bound)
template <int V, typename In, typename Op>
__global__ void __launch_bounds__(256) k_permute_lines(In in, const __grid_constant__ LineArgs a, Op op) {
    const int per = 256 / a.tpl, lane = threadIdx.x % a.tpl;
    const long long units = a.nlines * a.nseg;
    for (long long u = blockIdx.x * (long long)per + threadIdx.x / a.tpl; u < units; u += (long long)gridDim.x * per) {
        // (32-bit division where it suffices)
        const long long line = a.nseg == 1 ? u : u <= 0xffffffffLL ? (long long)((unsigned)u / (unsigned)a.nseg) : u / a.nseg;
        const long long x0 = (u - line * a.nseg) * a.seg, x1 = min(a.len, x0 + a.seg);
        long long r = line, off = 0;
        for (int j = a.nd - 1; j >= 0; --j) {
            const long long d = a.dout[j], q = r <= 0xffffffffLL ? (long long)((unsigned)r / (unsigned)d) : r / d;
            off += (r - q * d) * a.sin[j];
            r = q;
        }
        const long long ad = op.addr(line * a.len);
        constexpr int U = V == 4 ? 2 : 4;
        for (long long x = x0 + V * lane; x < x1; x += U * V * a.tpl) {
            decltype(in(0)) v[U][V];
#pragma unroll
            for (int w = 0; w < U; ++w)
                if (x + w * V * a.tpl < x1)
#pragma unroll
                    for (int e = 0; e < V; ++e) v[w][e] = in(off + x + w * V * a.tpl + e);
#pragma unroll
            for (int w = 0; w < U; ++w)
                if (x + w * V * a.tpl < x1) op.template put_n<V>(ad + x + w * V * a.tpl, v[w]);
        }
        if (x1 == a.len) op.finish(line * a.len, a.len, ad, lane, a.tpl);
    }
}

template <typename In, typename Op>
__global__ void __launch_bounds__(256) k_permute_tiled(In in, TileArgs a, Op op) {
    __shared__ decltype(in(0)) tile[32][33];
    for (long long b = blockIdx.x; b < a.nblocks; b += gridDim.x) {
        long long t = b;
        const long long tx = t % a.ntx;
        t /= a.ntx;
        const long long ty = t % a.nty;
        t /= a.nty;
        long long in_off = 0, out_lin = 0;
        for (int j = a.nrest - 1; j >= 0; --j) {
            const long long cj = t % a.rdim[j];
            t /= a.rdim[j];
            in_off += cj * a.rsin[j];
            out_lin += cj * a.rsout[j];
        }
        const long long x0 = tx * 32, y0 = ty * 32;
        for (int i = threadIdx.y; i < 32; i += 8) {
            const long long x = x0 + i, y = y0 + threadIdx.x;
            if (x < a.nx && y < a.ny) tile[threadIdx.x][i] = in(in_off + x * a.sx_in + y);
        }
        __syncthreads();
        for (int i = threadIdx.y; i < 32; i += 8) {
            const long long y = y0 + i, x = x0 + threadIdx.x;
            if (y < a.ny && x < a.nx) {
                // the row's 32 x values share one output row (x is the innermost output axis)
                const long long ad = op.addr(out_lin + y * a.sy_out + x0);
                op.put(ad + threadIdx.x, tile[i][threadIdx.x]);
            }
        }
        __syncthreads();
    }
}

// zero the K padding columns of split planes [rows][Kp]
__global__ void k_zero_pad(__nv_bfloat16* __restrict__ o0, __nv_bfloat16* __restrict__ o1, __nv_bfloat16* __restrict__ o2,
                           long long rows, long long K, long long Kp) {
    const long long w = Kp - K, n = rows * w;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const long long r = i / w, k = K + (i - r * w);
        o0[r * Kp + k] = __double2bfloat16(0.0);
        o1[r * Kp + k] = __double2bfloat16(0.0);
        if (o2) o2[r * Kp + k] = __double2bfloat16(0.0);
    }
}

inline int grid_for(long long n) {
    long long g = (n + 255) / 256;
    return (int)std::min<long long>(std::max<long long>(g, 1), 152LL * 32);
}

// ---- own GEMM kernels for the skinny contractions of the mixed sigma ----------------
// Row-major A [M][K] (lda), B [K][N] (ldb): FP64 operands rounded to FP32 in registers, FP32 products
// summed in FP32 over at most 64 terms, those partial sums accumulated in FP64 (the FP32-accurate
// class).  Each kernel writes its K slice's partial result P[slice][m][n]; k_reduce_slices finishes
// C = alpha sum_slices P + beta C.

// Both are bound by reading the large operand, as far as enough of its bytes are in flight: blocks of 128
// threads waste less of an SM's registers and of the last wave than ones of 256 (one to three resident
// blocks), and the FP64 adds (two a cycle and SM) are kept to one a result and 64 terms.
// Measured, the products of a 4-vector EA sigma with the coupling block (blocks of 256 -> 128, wider loads
// in flight, folded sums): 180 x 648,000 (467 MB) row 162 -> 96 us, column 138 -> 88 us (5 TB/s); 400 x
// 6,400,000 (10.2 GB) 2.2 -> 1.6 and 2.1 -> 1.5 ms (6.2 and 6.7 TB/s).  64 threads, 16 loads, 8 rows a block
// and more slices are no faster.
constexpr int SK_THREADS = 128;
constexpr int SK_CHUNK = 64;  // FP32 partial-sum length

// M <= MM rows of A (a few trial vectors): V consecutive columns of B per thread (4 where every row of B
// starts on a 16-byte boundary, N % 4 == 0: enough bytes in flight for the memory system), the A values
// of the current K chunk in shared memory; reads B once, coalesced along n.
template <int MM, int V, typename TB>
__global__ void __launch_bounds__(SK_THREADS, V == 4 && MM <= 4 && sizeof(TB) == 4 ? 5 : 1) k_skinny_m(int M, long long N, long long K, long long kslice,
                                                         const double* __restrict__ A, long long lda,
                                                         const TB* __restrict__ B, long long ldb,
                                                         double* __restrict__ P, double alpha, double beta) {
    __shared__ float As[MM][SK_THREADS];  // the A chunk, already rounded to FP32
    const long long n = (blockIdx.x * (long long)SK_THREADS + threadIdx.x) * V;
    const long long k0 = blockIdx.y * kslice, k1 = min(K, k0 + kslice);
    double acc[MM][V];
#pragma unroll
    for (int m = 0; m < MM; ++m)
#pragma unroll
        for (int e = 0; e < V; ++e) acc[m][e] = 0.0;
    for (long long kc = k0; kc < k1; kc += SK_THREADS) {
        const int kn = (int)min((long long)SK_THREADS, k1 - kc);
        __syncthreads();
        if (threadIdx.x < kn)
#pragma unroll
            for (int m = 0; m < MM; ++m) As[m][threadIdx.x] = (float)(m < M ? A[m * lda + kc + threadIdx.x] : 0.0);
        __syncthreads();
        if (n >= N) continue;
        const TB* b = B + kc * ldb + n;
        // U independent loads in flight per thread before their FMAs (the loop is bound by
        // memory latency otherwise)
        constexpr int U = V == 4 && sizeof(TB) == 8 ? 4 : 8;
        for (int k2 = 0; k2 < kn; k2 += SK_CHUNK) {
            float part[MM][V];
#pragma unroll
            for (int m = 0; m < MM; ++m)
#pragma unroll
                for (int e = 0; e < V; ++e) part[m][e] = 0.f;
            const int ke = min(kn, k2 + SK_CHUNK);
            for (int kk = k2; kk < ke; kk += U) {
                TB bv[U][V];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const TB* p = b + (long long)(kk + u < ke ? kk + u : ke - 1) * ldb;
                    if constexpr (V == 4 && sizeof(TB) == 4) {
                        *(float4*)bv[u] = *(const float4*)p;
                    } else if constexpr (V == 4) {
                        ((double2*)bv[u])[0] = ((const double2*)p)[0];
                        ((double2*)bv[u])[1] = ((const double2*)p)[1];
                    } else {
                        bv[u][0] = *p;
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int m = 0; m < MM; ++m) {
                        const float a = kk + u < ke ? As[m][kk + u] : 0.f;
#pragma unroll
                        for (int e = 0; e < V; ++e) part[m][e] = fmaf(a, (float)bv[u][e], part[m][e]);
                    }
            }
            const bool first = kc == k0 && k2 == 0;
            if (first) {
#pragma unroll
                for (int m = 0; m < MM; ++m)
#pragma unroll
                    for (int e = 0; e < V; ++e) acc[m][e] = (double)part[m][e];
            } else {
#pragma unroll
                for (int m = 0; m < MM; ++m)
#pragma unroll
                    for (int e = 0; e < V; ++e) acc[m][e] += (double)part[m][e];
            }
        }
    }
    if (n < N)
#pragma unroll
        for (int m = 0; m < MM; ++m)
            if (m < M)
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    double* p = P + ((long long)blockIdx.y * M + m) * N + n + e;
                    const double x = alpha == 1.0 ? acc[m][e] : alpha * acc[m][e];
                    *p = beta == 0.0 ? x : x + beta * *p;
                }
}

// N <= NN columns, B as [N][K]: a block takes RR rows of A and a K slice; threads stride over k (A and
// B read coalesced, B once for all RR rows), then a warp-shuffle and shared-memory reduction.
// V consecutive terms per thread at a time: 4 where every row starts on a 16-byte boundary (K % 4 == 0),
// which keeps enough bytes in flight for the memory system; else 1.
template <int NN, int V, typename TA>
__global__ void __launch_bounds__(SK_THREADS) k_skinny_n(long long M, int N, long long K, long long kslice,
                                                         const TA* __restrict__ A, long long lda,
                                                         const float* __restrict__ B, long long ldb,
                                                         double* __restrict__ P) {
    constexpr int RR = 4;
    constexpr int NV = NN == 1 ? RR : NN == 2 ? 2 * RR : NN <= 4 ? 4 * RR : 8 * RR;  // RR NN to a power of two
    __shared__ double red[SK_THREADS / 32][NV];
    const long long m0 = blockIdx.x * (long long)RR;
    const long long k0 = blockIdx.y * kslice, k1 = min(K, k0 + kslice);
    const TA* a[RR];  // rows past the last read the last one and are discarded
#pragma unroll
    for (int r = 0; r < RR; ++r) a[r] = A + min(m0 + r, M - 1) * lda;
    double acc[RR][NN];
#pragma unroll
    for (int r = 0; r < RR; ++r)
#pragma unroll
        for (int j = 0; j < NN; ++j) acc[r][j] = 0.0;
    // each thread takes SK_CHUNK of its terms per FP32 partial sum
    for (long long kb = k0; kb < k1; kb += (long long)SK_THREADS * SK_CHUNK) {
        float part[RR][NN];
#pragma unroll
        for (int r = 0; r < RR; ++r)
#pragma unroll
            for (int j = 0; j < NN; ++j) part[r][j] = 0.f;
        const long long ke = min(k1, kb + (long long)SK_THREADS * SK_CHUNK);
#pragma unroll 2
        for (long long k = kb + V * threadIdx.x; k < ke; k += V * SK_THREADS) {
            TA av[RR][V];
            float bv[NN][V];
#pragma unroll
            for (int r = 0; r < RR; ++r) {
                if constexpr (V == 4 && sizeof(TA) == 4) {
                    *(float4*)av[r] = *(const float4*)(a[r] + k);
                } else if constexpr (V == 4) {
                    ((double2*)av[r])[0] = ((const double2*)(a[r] + k))[0];
                    ((double2*)av[r])[1] = ((const double2*)(a[r] + k))[1];
                } else {
                    av[r][0] = a[r][k];
                }
            }
#pragma unroll
            for (int j = 0; j < NN; ++j)
            {
                const float* b = B + (j < N ? j : 0) * ldb + k;
                if constexpr (V == 4)
                    *(float4*)bv[j] = *(const float4*)b;
                else
                    bv[j][0] = *b;
            }
#pragma unroll
            for (int e = 0; e < V; ++e)
#pragma unroll
                for (int j = 0; j < NN; ++j) {
                    const float b = bv[j][e];
#pragma unroll
                    for (int r = 0; r < RR; ++r) part[r][j] = fmaf((float)av[r][e], b, part[r][j]);
                }
        }
#pragma unroll
        for (int r = 0; r < RR; ++r)
#pragma unroll
            for (int j = 0; j < NN; ++j) acc[r][j] += (double)part[r][j];
    }
    double val[NV];
#pragma unroll
    for (int x = 0; x < NV; ++x) val[x] = x < RR * NN ? acc[x / NN % RR][x % NN] : 0.0;
    const int lane = threadIdx.x & 31;
    warp_fold<NV>(val, lane);
    if (lane % (32 / NV) == 0) red[threadIdx.x >> 5][lane * NV / 32] = val[0];
    __syncthreads();
    if (threadIdx.x < RR * NN) {
        const int r = threadIdx.x / NN, j = threadIdx.x % NN;
        double x = 0.0;
        for (int w = 0; w < SK_THREADS / 32; ++w) x += red[w][threadIdx.x];
        if (m0 + r < M && j < N) P[((long long)blockIdx.y * M + m0 + r) * N + j] = x;
    }
}

// As k_reduce_slices for many slices: one warp per output element, lanes over slices,
// then a shuffle reduction.
template <typename Tp>
__global__ void k_reduce_slices_warp(int S, long long M, long long N, const Tp* __restrict__ P, double alpha,
                                     double beta, double* __restrict__ C, long long ldc) {
    const long long total = M * N;
    const int lane = threadIdx.x & 31;
    const long long warps = (long long)gridDim.x * blockDim.x / 32;
    for (long long x = (blockIdx.x * (long long)blockDim.x + threadIdx.x) / 32; x < total; x += warps) {
        double a = 0.0;
        for (int s2 = lane; s2 < S; s2 += 32) a += (double)P[s2 * total + x];
        for (int off = 16; off > 0; off >>= 1) a += __shfl_down_sync(0xffffffffu, a, off);
        if (lane == 0) {
            const long long m = x / N, n = x - m * N;
            double* cp = C + m * ldc + n;
            *cp = beta == 0.0 ? alpha * a : alpha * a + beta * *cp;
        }
    }
}

// C[m * ldc + n] = alpha sum_s P[s][m][n] + beta C[m * ldc + n]
__global__ void k_reduce_slices(int S, long long M, long long N, const double* __restrict__ P, double alpha, double beta,
                                double* __restrict__ C, long long ldc) {
    const long long total = M * N;
    for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < total; x += (long long)gridDim.x * blockDim.x) {
        double a = 0.0;
        for (int s2 = 0; s2 < S; ++s2) a += P[s2 * total + x];
        const long long m = x / N, n = x - m * N;
        double* cp = C + m * ldc + n;
        *cp = beta == 0.0 ? alpha * a : alpha * a + beta * *cp;
    }
}

}  // namespace

void own_gemm(Ctx& c, long long M, long long N, long long K, double alpha, const void* A, bool a32, const void* B, bool b32,
              double beta, double* C) {
    if (M <= 0 || N <= 0) return;
    if (K <= 0) {
        if (beta == 0.0)
            fill(c, M * N, 0.0, C);
        else if (beta != 1.0)
            axpby(c, M * N, 0.0, C, beta, C);
        return;
    }
    const long long target = 152LL * 8;  // blocks that fill the GPU several times over
    const long long kch = (K + SK_THREADS - 1) / SK_THREADS;
    Arena::Mark mk = c.arena.mark();
    int S = 1;
    double* P = nullptr;
    auto slices = [&](long long blocks) {
        S = (int)std::max<long long>(1, std::min<long long>({kch, (target + blocks - 1) / blocks, 512}));
        const long long ks = (kch + S - 1) / S * SK_THREADS;
        S = (int)((K + ks - 1) / ks);
        return ks;
    };
    if (M <= 8) {
        if (a32) throw Error(-1, "own_gemm: the small operand is FP64");
        const bool vec = N % 4 == 0 && (uintptr_t)B % 16 == 0 && N >= 4096;
        const long long cols = vec ? 4 * SK_THREADS : SK_THREADS, nbn = (N + cols - 1) / cols, ks = slices(nbn);
        P = S == 1 ? C : c.arena.dalloc((size_t)S * M * N);
        const double al = S == 1 ? alpha : 1.0, be = S == 1 ? beta : 0.0;
        const dim3 g((unsigned)nbn, (unsigned)S);
        switch ((int)M) {
#define SKM_GO(X, V, TB) k_skinny_m<X, V, TB><<<g, SK_THREADS, 0, c.stream>>>((int)M, N, K, ks, (const double*)A, K, (const TB*)B, N, P, al, be)
#define SKM(X)                                                       \
    case X:                                                          \
        if (b32) {                                                   \
            if (vec) SKM_GO(X, 4, float); else SKM_GO(X, 1, float);  \
        } else {                                                     \
            if (vec) SKM_GO(X, 4, double); else SKM_GO(X, 1, double); \
        }                                                            \
        break;
            SKM(1) SKM(2) SKM(3) SKM(4) SKM(5) SKM(6) SKM(7) SKM(8)
#undef SKM
#undef SKM_GO
        }
    } else if (N <= 8) {
        if (!b32) throw Error(-1, "own_gemm: the small operand is FP32");
        constexpr int RR = 4;
        const bool vec = K % 4 == 0 && (uintptr_t)A % 16 == 0 && (uintptr_t)B % 16 == 0;
        const long long mb = (M + RR - 1) / RR, ks = slices(mb);
        if (mb > 0x7fffffffLL) throw Error(-1, "own_gemm: too many rows");
        P = c.arena.dalloc((size_t)S * M * N);
        const dim3 g((unsigned)mb, (unsigned)S);
        switch ((int)N) {
#define SKN_GO(X, V, TA) k_skinny_n<X, V, TA><<<g, SK_THREADS, 0, c.stream>>>(M, (int)N, K, ks, (const TA*)A, K, (const float*)B, K, P)
#define SKN(X)                                                       \
    case X:                                                          \
        if (a32) {                                                   \
            if (vec) SKN_GO(X, 4, float); else SKN_GO(X, 1, float);  \
        } else {                                                     \
            if (vec) SKN_GO(X, 4, double); else SKN_GO(X, 1, double); \
        }                                                            \
        break;
            SKN(1) SKN(2) SKN(3) SKN(4) SKN(5) SKN(6) SKN(7) SKN(8)
#undef SKN
#undef SKN_GO
        }
    } else {
        throw Error(-1, "own_gemm: neither side is skinny");
    }
    ++c.kernels;
    ADC_CUDA(cudaGetLastError());
    if (P != C) {
        if (S >= 16)
            k_reduce_slices_warp<double><<<grid_for(32 * M * N), 256, 0, c.stream>>>(S, M, N, P, alpha, beta, C, N);
        else
            k_reduce_slices<<<grid_for(M * N), 256, 0, c.stream>>>(S, M, N, P, alpha, beta, C, N);
        ++c.kernels;
        ADC_CUDA(cudaGetLastError());
    }
    c.arena.release(mk);
}

// The tiled form applies when, after dropping unit axes, the output's innermost axis is
// strided in the input and both it and the input-contiguous axis are at least 8 long.
static bool tiled_args(const PermArgs& p, TileArgs& t) {
    long long d[kMaxDim], si[kMaxDim];
    int nd = 0;
    for (int j = 0; j < p.nd; ++j)
        if (p.dout[j] > 1) {
            d[nd] = p.dout[j];
            si[nd] = p.sin[j];
            ++nd;
        }
    if (nd < 2 || si[nd - 1] == 1) return false;
    int jy = -1;
    for (int j = 0; j < nd - 1; ++j)
        if (si[j] == 1) jy = j;
    if (jy < 0 || d[jy] < 8 || d[nd - 1] < 8) return false;
    long long so[kMaxDim], acc = 1;
    for (int j = nd - 1; j >= 0; --j) {
        so[j] = acc;
        acc *= d[j];
    }
    t.nrest = 0;
    long long rest = 1;
    for (int j = 0; j < nd - 1; ++j) {
        if (j == jy) continue;
        t.rdim[t.nrest] = d[j];
        t.rsin[t.nrest] = si[j];
        t.rsout[t.nrest] = so[j];
        ++t.nrest;
        rest *= d[j];
    }
    t.nx = d[nd - 1];
    t.sx_in = si[nd - 1];
    t.ny = d[jy];
    t.sy_out = so[jy];
    t.ntx = (t.nx + 31) / 32;
    t.nty = (t.ny + 31) / 32;
    t.nblocks = t.ntx * t.nty * rest;
    return true;
}

template <typename In, typename Op>
static void launch_tiled(Ctx& c, const In& in, const TileArgs& t, const Op& op) {
    const long long g = std::min<long long>(t.nblocks, 152LL * 16);
    k_permute_tiled<In, Op><<<(unsigned)g, dim3(32, 8), 0, c.stream>>>(in, t, op);
    ++c.kernels;
    ADC_CUDA(cudaGetLastError());
}

static PermArgs perm_args(const Shape& s, const int* perm, long long& total) {
    PermArgs a;
    a.nd = s.nd;
    long long st[kMaxDim];
    long long acc = 1;
    total = 1;
    for (int j = s.nd - 1; j >= 0; --j) {
        st[j] = acc;
        acc *= s.d[j];
    }
    for (int j = 0; j < s.nd; ++j) {
        a.dout[j] = s.d[perm[j]];
        a.sin[j] = st[perm[j]];
        total *= a.dout[j];
    }
    return a;
}

// The line form applies when the output's fastest axis is contiguous in the input (axes that are
// neighbours on both sides are merged first, within a row of `unit` elements if it is not 0) and at
// least 8 long.
static bool line_args(const PermArgs& p, long long unit, LineArgs& t) {
    long long d[kMaxDim], si[kMaxDim];
    int nd = 0;
    for (int j = 0; j < p.nd; ++j)
        if (p.dout[j] > 1) {
            d[nd] = p.dout[j];
            si[nd] = p.sin[j];
            ++nd;
        }
    if (nd == 0 || si[nd - 1] != 1) return false;
    t.len = d[--nd];
    while (nd > 0 && si[nd - 1] == t.len && (unit == 0 || unit % (t.len * d[nd - 1]) == 0)) t.len *= d[--nd];
    if (t.len < 8 || (unit && unit % t.len)) return false;
    t.nd = nd;
    t.nlines = 1;
    for (int j = 0; j < nd; ++j) {
        t.dout[j] = d[j];
        t.sin[j] = si[j];
        t.nlines *= d[j];
    }
    // segments of at most 1024 elements, of 256 when that still leaves the chip idle
    t.seg = std::min<long long>(1024, (t.len + 3) / 4 * 4);
    if (t.nlines * ((t.len + t.seg - 1) / t.seg) < 2048) t.seg = std::min<long long>(t.seg, 256);
    const long long ns = (t.len + t.seg - 1) / t.seg;
    if (ns > 0x7fffffffLL) return false;
    t.nseg = (int)ns;
    t.tpl = 8;
    while (t.tpl < 256 && t.tpl * 8 < t.seg) t.tpl *= 2;
    return true;
}

template <typename In, typename Op>
static void launch_lines(Ctx& c, const In& in, const LineArgs& t, const Op& op) {
    const long long per = 256 / t.tpl, g = std::min<long long>((t.nlines * t.nseg + per - 1) / per, 152LL * 32);
    if (t.len % 4 == 0)
        k_permute_lines<4, In, Op><<<(unsigned)g, 256, 0, c.stream>>>(in, t, op);
    else
        k_permute_lines<1, In, Op><<<(unsigned)g, 256, 0, c.stream>>>(in, t, op);
    ++c.kernels;
    ADC_CUDA(cudaGetLastError());
}

template <typename In, typename Tout>
static void permute_in(Ctx& c, const In& in, const Shape& s, const int* perm, Tout* out, double alpha, double beta) {
    long long total;
    PermArgs a = perm_args(s, perm, total);
    if (total == 0) return;
    TileArgs t;
    if (tiled_args(a, t)) {
        launch_tiled(c, in, t, OpAxpby<Tout>{out, alpha, beta});
        return;
    }
    LineArgs ln;
    if (line_args(a, 0, ln)) {
        launch_lines(c, in, ln, OpAxpby<Tout>{out, alpha, beta});
        return;
    }
    if (total <= 0xffffffffLL)  // every offset is below total
        permute_kernel<unsigned, In, Tout><<<grid_for(total), 256, 0, c.stream>>>(in, out, a, total, alpha, beta);
    else
        permute_kernel<long long, In, Tout><<<grid_for(total), 256, 0, c.stream>>>(in, out, a, total, alpha, beta);
    ++c.kernels;
    ADC_CUDA(cudaGetLastError());
}

void permute(Ctx& c, const double* in, const Shape& s, const int* perm, double* out, double alpha, double beta) {
    permute_in(c, Plain<double>{in}, s, perm, out, alpha, beta);
}

template <typename Tin>
static void permute_sum_t(Ctx& c, const Tin* in, int S, const Shape& s, const int* perm, void* out, bool out32, double alpha,
                          double beta) {
    long long n = 1;
    for (int j = 0; j < s.nd; ++j) n *= s.d[j];
    if (S == 1) {
        if (out32)
            permute_in(c, Plain<Tin>{in}, s, perm, (float*)out, alpha, beta);
        else
            permute_in(c, Plain<Tin>{in}, s, perm, (double*)out, alpha, beta);
        return;
    }
    Arena::Mark mk = c.arena.mark();
    if (S >= 16) {
        // many slices are summed by a warp per element first
        double* sum = c.arena.dalloc((size_t)n);
        k_reduce_slices_warp<Tin><<<grid_for(32 * n), 256, 0, c.stream>>>(S, 1, n, in, 1.0, 0.0, sum, n);
        ++c.kernels;
        ADC_CUDA(cudaGetLastError());
        permute_sum_t(c, (const double*)sum, 1, s, perm, out, out32, alpha, beta);
        c.arena.release(mk);
        return;
    }
    if (out32)
        permute_in(c, SumOf<Tin>{in, S, n}, s, perm, (float*)out, alpha, beta);
    else
        permute_in(c, SumOf<Tin>{in, S, n}, s, perm, (double*)out, alpha, beta);
}
void permute_sum(Ctx& c, const float* in, int S, const Shape& s, const int* perm, void* out, bool out32, double alpha,
                 double beta) {
    permute_sum_t(c, in, S, s, perm, out, out32, alpha, beta);
}
void permute_sum(Ctx& c, const double* in, int S, const Shape& s, const int* perm, void* out, bool out32, double alpha,
                 double beta) {
    permute_sum_t(c, in, S, s, perm, out, out32, alpha, beta);
}

template <typename Tin>
static void split_planes_t(Ctx& c, const Tin* in, const PermArgs& a, long long rows, long long K, long long Kp,
                           void* const* out, int planes) {
    TileArgs t;
    __nv_bfloat16 *o0 = (__nv_bfloat16*)out[0], *o1 = (__nv_bfloat16*)out[1];
    __nv_bfloat16* o2 = planes == 3 ? (__nv_bfloat16*)out[2] : nullptr;
    if (tiled_args(a, t)) {
        launch_tiled(c, Plain<Tin>{in}, t, OpPlanes{o0, o1, o2, K, Kp});
        if (Kp > K) {
            k_zero_pad<<<grid_for(rows * (Kp - K)), 256, 0, c.stream>>>(o0, o1, o2, rows, K, Kp);
            ++c.kernels;
            ADC_CUDA(cudaGetLastError());
        }
        return;
    }
    LineArgs ln;
    if (line_args(a, K, ln)) {
        launch_lines(c, Plain<Tin>{in}, ln, OpPlanes{o0, o1, o2, K, Kp});
        return;
    }
    // 32-bit coordinates when the output index fits (every input offset is below rows * K)
    if (rows * Kp <= 0xffffffffLL)
        permute_split_kernel<unsigned, Tin><<<grid_for(rows * Kp), 256, 0, c.stream>>>(in, o0, o1, o2, a, rows, K, Kp);
    else
        permute_split_kernel<long long, Tin><<<grid_for(rows * Kp), 256, 0, c.stream>>>(in, o0, o1, o2, a, rows, K, Kp);
    ++c.kernels;
    ADC_CUDA(cudaGetLastError());
}

void split_planes(Ctx& c, const double* in, const Shape& s, const int* perm, long long rows, long long K, long long Kp,
                  void* const* out, bool in32, int planes) {
    long long total;
    PermArgs a = perm_args(s, perm, total);
    if (total != rows * K) throw Error(-1, "split_planes: shape mismatch");
    if (rows * Kp == 0) return;
    if (in32)
        split_planes_t(c, (const float*)in, a, rows, K, Kp, out, planes);
    else
        split_planes_t(c, in, a, rows, K, Kp, out, planes);
}

void permute_any(Ctx& c, const void* in, bool in32, const Shape& s, const int* perm, void* out, bool out32,
                 double alpha, double beta) {
    const Plain<double> d{(const double*)in};
    const Plain<float> f{(const float*)in};
    if (!in32 && !out32)
        permute_in(c, d, s, perm, (double*)out, alpha, beta);
    else if (in32 && out32)
        permute_in(c, f, s, perm, (float*)out, alpha, beta);
    else if (in32)
        permute_in(c, f, s, perm, (double*)out, alpha, beta);
    else
        permute_in(c, d, s, perm, (float*)out, alpha, beta);
}

void axpby(Ctx& c, long long n, double alpha, const double* x, double beta, double* y) {
    if (n <= 0) return;
    axpby_kernel<<<grid_for(n), 256, 0, c.stream>>>(n, alpha, x, beta, y);
    ++c.kernels;
    ADC_CUDA(cudaGetLastError());
}

void fill(Ctx& c, long long n, double v, double* y) {
    if (n <= 0) return;
    fill_kernel<<<grid_for(n), 256, 0, c.stream>>>(n, v, y);
    ++c.kernels;
    ADC_CUDA(cudaGetLastError());
}

void gemm(Ctx& c, bool ta, bool tb, long long M, long long N, long long K, double alpha, const double* A, long long lda,
          long long sA, const double* B, long long ldb, long long sB, double beta, double* C, long long ldc,
          long long sC, long long batch) {
    if (M <= 0 || N <= 0 || batch <= 0) return;
    if (K <= 0) {
        // C = beta C
        if (ldc == N && (batch == 1 || sC == M * N)) {
            if (beta == 0.0)
                fill(c, M * N * batch, 0.0, C);
            else if (beta != 1.0)
                axpby(c, M * N * batch, 0.0, C, beta, C);
            return;
        }
        throw Error(-1, "gemm: K == 0 with strided C");
    }
    // row-major C = op(A) op(B)  <=>  column-major C^T = op(B)^T op(A)^T
    cublasOperation_t oa = ta ? CUBLAS_OP_T : CUBLAS_OP_N;
    cublasOperation_t ob = tb ? CUBLAS_OP_T : CUBLAS_OP_N;
    if (batch == 1) {
        ADC_BLAS(cublasDgemm(c.blas, ob, oa, (int)N, (int)M, (int)K, &alpha, B, (int)ldb, A, (int)lda, &beta, C, (int)ldc));
    } else {
        ADC_BLAS(cublasDgemmStridedBatched(c.blas, ob, oa, (int)N, (int)M, (int)K, &alpha, B, (int)ldb, sB, A, (int)lda,
                                           sA, &beta, C, (int)ldc, sC, (int)batch));
    }
}

namespace {

struct Spec {
    std::string a, b, c;
};

Spec parse(const char* spec) {
    std::string s(spec);
    size_t comma = s.find(','), arrow = s.find("->");
    if (comma == std::string::npos || arrow == std::string::npos || comma > arrow)
        throw Error(-1, std::string("einsum: bad spec ") + spec);
    return {s.substr(0, comma), s.substr(comma + 1, arrow - comma - 1), s.substr(arrow + 2)};
}

bool has(const std::string& s, char x) { return s.find(x) != std::string::npos; }

// permute src (letters ls, dims) into the letter order lt; returns pointer (src if identity)
// (an FP32 operand is always converted into an FP64 copy)
const double* to_order(Ctx& c, const double* src, const std::string& ls, const std::map<char, long long>& dim,
                       const std::string& lt, bool f32 = false) {
    if (ls == lt && !f32) return src;
    Shape sh;
    sh.nd = (int)ls.size();
    long long n = 1;
    for (int j = 0; j < sh.nd; ++j) {
        sh.d[j] = dim.at(ls[j]);
        n *= sh.d[j];
    }
    int perm[kMaxDim];
    for (int j = 0; j < sh.nd; ++j) perm[j] = (int)ls.find(lt[j]);
    double* dst = c.arena.dalloc(n);
    permute_any(c, src, f32, sh, perm, dst, false, 1.0, 0.0);
    return dst;
}

}  // namespace

// FP32-accurate contraction: operands permuted and rounded to FP32, GEMM with
// BF16x9 emulation (falls back to plain FP32 if the library lacks it), result
// permuted and accumulated into the FP64 output.
static void einsum_fp32(Ctx& c, const std::string& la, const std::string& lb, const std::string& lc,
                        std::map<char, long long>& dim, const std::string& batch, const std::string& fa,
                        const std::string& fb, const std::string& con, double alpha, const T& A, const T& B,
                        double beta, void* C, bool c32) {
    auto prod = [&](const std::string& l) {
        long long p = 1;
        for (char x : l) p *= dim[x];
        return p;
    };
    long long nb = prod(batch), M = prod(fa), N = prod(fb), K = prod(con);
    auto conv = [&](const T& X, const std::string& ls, const std::string& lt) {
        // an FP32 operand already in GEMM order is used in place
        if (X.f32 && ls == lt) return (const float*)X.p;
        Shape sh;
        sh.nd = (int)ls.size();
        long long n = 1;
        for (int j = 0; j < sh.nd; ++j) {
            sh.d[j] = dim.at(ls[j]);
            n *= sh.d[j];
        }
        int perm[kMaxDim];
        std::string key;
        for (int j = 0; j < sh.nd; ++j) {
            perm[j] = (int)ls.find(lt[j]);
            key += (char)('0' + perm[j]);
            key += ':';
            key += std::to_string(sh.d[j]);
            key += ',';
        }
        float* dst;
        if (X.constant && (size_t)n * sizeof(float) <= c.cache_max_bytes) {
            auto it = c.f32cache.find({X.p, key});
            if (it != c.f32cache.end()) return (const float*)it->second;
            if (c.capturing) throw Error(-3, "operand cache miss during stream capture");
            dst = (float*)dev_alloc(n * sizeof(float), c.stream);
            c.f32cache[{X.p, key}] = dst;
        } else {
            dst = (float*)c.arena.alloc(n * sizeof(float));
        }
        permute_any(c, X.p, X.f32, sh, perm, dst, true, 1.0, 0.0);
        return (const float*)dst;
    };
    const float* A32 = conv(A, la, batch + fa + con);
    const float* B32 = conv(B, lb, batch + con + fb);
    const std::string tord = batch + fa + fb;
    // an FP32 output in the GEMM's order is written by the GEMM itself (C = alpha AB + beta C)
    const bool direct = c32 && tord == lc;
    float* T32 = direct ? (float*)C : (float*)c.arena.alloc(nb * M * N * sizeof(float));
    const float one = direct ? (float)alpha : 1.0f, zero = direct ? (float)beta : 0.0f;
    // row-major T[M][N] = A[M][K] B[K][N]  <=>  column-major T^T = B^T A^T
    auto run = [&](cublasComputeType_t ct) {
        return cublasGemmStridedBatchedEx(c.blas, CUBLAS_OP_N, CUBLAS_OP_N, (int)N, (int)M, (int)K, &one, B32, CUDA_R_32F,
                                          (int)N, K * N, A32, CUDA_R_32F, (int)K, M * K, &zero, T32, CUDA_R_32F, (int)N,
                                          M * N, (int)nb, ct, CUBLAS_GEMM_DEFAULT);
    };
    if (c.emulation_ok != 0) {
        cublasStatus_t st = run(CUBLAS_COMPUTE_32F_EMULATED_16BFX9);
        if (st == CUBLAS_STATUS_SUCCESS) {
            c.emulation_ok = 1;
        } else if (c.emulation_ok == -1 && (st == CUBLAS_STATUS_NOT_SUPPORTED || st == CUBLAS_STATUS_INVALID_VALUE)) {
            c.emulation_ok = 0;
            ADC_BLAS(run(CUBLAS_COMPUTE_32F));
        } else {
            ADC_BLAS(st);
        }
    } else {
        ADC_BLAS(run(CUBLAS_COMPUTE_32F));
    }
    if (direct) return;
    Shape sh;
    sh.nd = (int)tord.size();
    for (int j = 0; j < sh.nd; ++j) sh.d[j] = dim[tord[j]];
    int perm[kMaxDim];
    for (int j = 0; j < sh.nd; ++j) perm[j] = (int)tord.find(lc[j]);
    permute_any(c, T32, true, sh, perm, C, c32, alpha, beta);
}

// Tensor-core contraction (gemm_mode 2): operands permuted into K-major GEMM
// order and split into two BF16 planes (constant operands once, cached), the
// tcgen05 split-BF16 GEMM into FP32 results (one per K slice), whose FP64 sum is permuted and
// accumulated into the output in one pass.
static void einsum_tc(Ctx& c, const std::string& la, const std::string& lb, const std::string& lc,
                      std::map<char, long long>& dim, const std::string& fa, const std::string& fb, const std::string& con,
                      double alpha, const T& A, const T& B, double beta, void* C, bool c32) {
    auto prod = [&](const std::string& l) {
        long long p = 1;
        for (char x : l) p *= dim[x];
        return p;
    };
    const long long M = prod(fa), N = prod(fb), K = prod(con), Kp = (K + 7) / 8 * 8;
    auto planes_of = [&](const T& X, const std::string& ls, const std::string& lt, long long rows) {
        Shape sh;
        sh.nd = (int)ls.size();
        for (int j = 0; j < sh.nd; ++j) sh.d[j] = dim.at(ls[j]);
        int perm[kMaxDim];
        std::string key = "bf16x2:";
        for (int j = 0; j < sh.nd; ++j) {
            perm[j] = (int)ls.find(lt[j]);
            key += (char)('0' + perm[j]);
            key += ':';
            key += std::to_string(sh.d[j]);
            key += ',';
        }
        key += std::to_string(K);
        void* base = nullptr;
        if (X.constant && (size_t)(2 * rows * Kp * 2) <= c.cache_max_bytes) {
            auto it = c.bf16cache.find({X.p, key});
            if (it != c.bf16cache.end()) return it->second;
            if (c.capturing) throw Error(-3, "operand cache miss during stream capture");
            base = dev_alloc(2 * rows * Kp * 2, c.stream);
            c.bf16cache[{X.p, key}] = base;
        } else {
            base = c.arena.alloc(2 * rows * Kp * 2);
        }
        void* out[2] = {base, (char*)base + rows * Kp * 2};
        split_planes(c, X.p, sh, perm, rows, K, Kp, out, X.f32);
        return base;
    };
    void* pa = planes_of(A, la, fa + con, M);
    void* pb = planes_of(B, lb, fb + con, N);
    if (!c.d_err) {
        if (c.capturing) throw Error(-3, "error flag allocation during stream capture");
        c.d_err = (int*)dev_alloc(sizeof(int), c.stream);
        ADC_CUDA(cudaMemsetAsync(c.d_err, 0, sizeof(int), c.stream));
    }
    const void* A2[2] = {pa, (const char*)pa + M * Kp * 2};
    const void* B2[2] = {pb, (const char*)pb + N * Kp * 2};
    int S = 1;
    const std::string tord = fa + fb;
    // an FP32 output in the GEMM's order takes the one slice's result itself
    float* direct = c32 && tord == lc && alpha == 1.0 && beta == 0.0 ? (float*)C : nullptr;
    const float* T = tc_gemm(c, A2, B2, M, N, Kp, 2.0 * M * N * K, S, direct);
    if (T == direct) return;
    Shape sh;
    sh.nd = (int)tord.size();
    for (int j = 0; j < sh.nd; ++j) sh.d[j] = dim[tord[j]];
    int perm[kMaxDim];
    for (int j = 0; j < sh.nd; ++j) perm[j] = (int)tord.find(lc[j]);
    permute_sum(c, T, S, sh, perm, C, c32, alpha, beta);
}

// FP64 contraction (gemm64 on the tensor cores, small64 below its sizes): the operands are read and
// the result is written through their strides; K slices are summed by the permute that puts them in
// place.
static void einsum_64(Ctx& c, const std::string& la, const std::string& lb, const std::string& lc,
                      std::map<char, long long>& dim, const std::string& fa, const std::string& fb, const std::string& con,
                      double alpha, const T& A, const T& B, double beta, void* C, bool c32) {
    auto strides = [&](const std::string& l) {
        std::map<char, long long> st;
        long long acc = 1;
        for (int j = (int)l.size() - 1; j >= 0; --j) {
            st[l[j]] = acc;
            acc *= dim[l[j]];
        }
        return st;
    };
    auto operand = [&](const T& X, const std::string& l, const std::string& rows) {
        Operand64 o;
        o.p = X.p;
        o.f32 = X.f32;
        const auto st = strides(l);
        for (char x : rows) o.row_axis(dim[x], st.at(x));
        for (char x : con) o.k_axis(dim[x], st.at(x));
        if (o.nk == 0) o.k_axis(1, 1);
        return o;
    };
    Operand64 a = operand(A, la, fa), b = operand(B, lb, fb);
    if (a.rows == 0 || b.rows == 0) return;  // nothing to write
    const bool tensor = gemm64_fits(a.rows, b.rows, a.K);
    // the 128-row axis takes the longer side when the other would leave it mostly empty
    // (small64: the longer side on the grid's x axis)
    const bool swap = tensor ? a.rows < 64 && b.rows > a.rows : a.rows > b.rows;
    // digits of a constant operand, kept while there is room
    Digits64 da, db;
    auto kept = [&](const T& X, const Operand64& o, const std::string& l, const std::string& rows, Digits64& d) {
        if (!tensor || !X.constant || (c.cache64_bytes == 0 && c.cache64.empty())) return false;
        const size_t bytes = digits64_bytes(o.rows, o.K);
        std::string key = l + ">" + rows + "," + con;
        for (char x : l) key += ":" + std::to_string(dim[x]);
        auto it = c.cache64.find({X.p, key});
        const bool known = it != c.cache64.end();
        if (!known || !it->second->mem[0]) {
            if (c.capturing || (!known && bytes > c.cache64_bytes)) return false;
            // (no other memory is given up for them: without room they are made in scratch)
            void* buf = nullptr;
            if (dev_malloc_raw(&buf, bytes, c.stream) != cudaSuccess) {
                cudaGetLastError();
                return false;
            }
            if (!known) {
                c.cache64_bytes -= bytes;
                it = c.cache64.emplace(std::make_pair((const void*)X.p, key), std::make_unique<Reclaimable>()).first;
                it->second->call = &c.call;
            }
            it->second->hold(buf, nullptr, ReclaimPin(c.call, c.stream));
            d = digits64_in(buf, o.rows, o.K);
            digitise64(c, &o, &d, 1);
            return true;
        }
        d = digits64_in(it->second->mem[0], o.rows, o.K);
        return true;
    };
    const bool ka = kept(A, a, la, fa, da), kb = kept(B, b, lb, fb, db);
    const std::string rows = swap ? fb : fa, cols = swap ? fa : fb;
    Out64 out;
    if (!c32) {
        out.p = (double*)C;
        out.alpha = alpha;
        out.beta = beta;
        const auto st = strides(lc);
        for (char x : rows) out.row_axis(dim[x], st.at(x));
        for (char x : cols) out.col_axis(dim[x], st.at(x));
    }
    int S = 1;
    const double* Tm = !tensor ? (swap ? small64(c, b, a, out, S) : small64(c, a, b, out, S))
                       : swap  ? gemm64(c, b, kb ? &db : nullptr, a, ka ? &da : nullptr, out, S)
                               : gemm64(c, a, ka ? &da : nullptr, b, kb ? &db : nullptr, out, S);
    if (!Tm) return;
    const std::string tord = rows + cols;
    Shape sh;
    sh.nd = (int)tord.size();
    int perm[kMaxDim];
    for (int j = 0; j < sh.nd; ++j) {
        sh.d[j] = dim[tord[j]];
        perm[j] = (int)tord.find(lc[j]);
    }
    permute_sum(c, Tm, S, sh, perm, C, c32, alpha, beta);
}

static void einsum_core(Ctx& c, const char* specstr, double alpha, const T& A, const T& B, double beta, void* C, bool c32,
                        const std::vector<long long>& cdims) {
    Spec sp = parse(specstr);
    if (sp.a.size() != A.dims.size() || sp.b.size() != B.dims.size() || sp.c.size() != cdims.size())
        throw Error(-1, std::string("einsum: rank mismatch in ") + specstr);
    std::map<char, long long> dim;
    auto put = [&](const std::string& l, const std::vector<long long>& d) {
        for (size_t j = 0; j < l.size(); ++j) {
            auto it = dim.find(l[j]);
            if (it != dim.end() && it->second != d[j])
                throw Error(-1, std::string("einsum: dimension mismatch in ") + specstr);
            dim[l[j]] = d[j];
        }
    };
    put(sp.a, A.dims);
    put(sp.b, B.dims);
    put(sp.c, cdims);
    std::string batch, fa, fb, con;
    for (char x : sp.c) {
        bool ia = has(sp.a, x), ib = has(sp.b, x);
        if (ia && ib)
            batch += x;
        else if (ia)
            fa += x;
        else if (ib)
            fb += x;
        else
            throw Error(-1, std::string("einsum: output index not in inputs: ") + specstr);
    }
    for (char x : sp.a) {
        if (has(sp.c, x)) continue;
        if (!has(sp.b, x)) throw Error(-1, std::string("einsum: summed index in one operand only: ") + specstr);
        con += x;
    }
    for (char x : sp.b)
        if (!has(sp.c, x) && !has(sp.a, x)) throw Error(-1, std::string("einsum: summed index in one operand only: ") + specstr);
    auto prod = [&](const std::string& l) {
        long long p = 1;
        for (char x : l) p *= dim[x];
        return p;
    };
    long long nb = prod(batch), M = prod(fa), N = prod(fb), K = prod(con);
    Arena::Mark mk = c.arena.mark();
    if (c.gemm_mode == 2 && nb == 1) {
        // the mixed sigma: tensor cores for the large contractions, own kernels for the rest
        const bool big = 2.0 * M * N * K >= c.fp32_min_flops;
        // few-vector shapes: the own bandwidth kernels read the large operand once, in place when
        // it is already in their order ([K][N] for M <= 8, [M][K] for N <= 8);
        // otherwise the tensor cores take them when the large operand is a constant of the
        // handle (its split planes are cached once, the permuted FP64 copy would be made per call)
        const bool skinny = std::min(M, N) <= 8;
        const bool big_const = M <= 8 ? B.constant : A.constant;
        const bool big_in_place = M <= 8 ? sp.b == con + fb : sp.a == fa + con;
        if (big && tc_gemm_fits(M, N, K) && (!skinny || (big_const && !big_in_place))) {
            einsum_tc(c, sp.a, sp.b, sp.c, dim, fa, fb, con, alpha, A, B, beta, C, c32);
        } else if (!big || !skinny) {
            einsum_64(c, sp.a, sp.b, sp.c, dim, fa, fb, con, alpha, A, B, beta, C, c32);
        } else {
            // the large operand is read in place, also as FP32, when it is in the kernels' order
            const std::string oa = fa + con, ob = M <= 8 ? con + fb : fb + con;
            const bool a32 = A.f32 && M > 8 && sp.a == oa, b32 = M > 8 || (B.f32 && sp.b == ob);
            const double* Ap = a32 ? A.p : to_order(c, A.p, sp.a, dim, oa, A.f32);
            const void* Bp;
            if (M > 8 && !(B.f32 && sp.b == ob)) {
                // the few columns rounded to FP32 once (the kernel would do it for every four rows)
                Shape bs;
                bs.nd = (int)sp.b.size();
                int bp[kMaxDim];
                for (int j = 0; j < bs.nd; ++j) {
                    bs.d[j] = dim[sp.b[j]];
                    bp[j] = (int)sp.b.find(ob[j]);
                }
                float* f = (float*)c.arena.alloc((size_t)(K * N) * sizeof(float));
                permute_any(c, B.p, B.f32, bs, bp, f, true, 1.0, 0.0);
                Bp = f;
            } else {
                Bp = b32 ? B.p : to_order(c, B.p, sp.b, dim, ob, B.f32);
            }
            const std::string tord = fa + fb;
            if (tord == sp.c && !c32) {
                own_gemm(c, M, N, K, alpha, Ap, a32, Bp, b32, beta, (double*)C);
            } else {
                double* Tm = c.arena.dalloc((size_t)(M * N));
                own_gemm(c, M, N, K, 1.0, Ap, a32, Bp, b32, 0.0, Tm);
                Shape sh;
                sh.nd = (int)tord.size();
                for (int j = 0; j < sh.nd; ++j) sh.d[j] = dim[tord[j]];
                int perm[kMaxDim];
                for (int j = 0; j < sh.nd; ++j) perm[j] = (int)tord.find(sp.c[j]);
                permute_any(c, Tm, false, sh, perm, C, c32, alpha, beta);
            }
        }
        c.arena.release(mk);
        return;
    }
    if (c.gemm_mode >= 1 && 2.0 * nb * M * N * K >= c.fp32_min_flops) {
        einsum_fp32(c, sp.a, sp.b, sp.c, dim, batch, fa, fb, con, alpha, A, B, beta, C, c32);
        c.arena.release(mk);
        return;
    }
    if (nb == 1 && K > 0 && (gemm64_fits(M, N, K) || (std::min(M, N) < 500000 && std::max(M, N) < (1LL << 31) && K < (1LL << 30)))) {
        einsum_64(c, sp.a, sp.b, sp.c, dim, fa, fb, con, alpha, A, B, beta, C, c32);
        c.arena.release(mk);
        return;
    }
    const double* Ap = to_order(c, A.p, sp.a, dim, batch + fa + con, A.f32);
    const double* Bp = to_order(c, B.p, sp.b, dim, batch + con + fb, B.f32);
    std::string tord = batch + fa + fb;
    if (tord == sp.c && !c32) {
        gemm(c, false, false, M, N, K, alpha, Ap, K, M * K, Bp, N, K * N, beta, (double*)C, N, M * N, nb);
    } else {
        double* Tm = c.arena.dalloc((size_t)(nb * M * N));
        gemm(c, false, false, M, N, K, 1.0, Ap, K, M * K, Bp, N, K * N, 0.0, Tm, N, M * N, nb);
        Shape sh;
        sh.nd = (int)tord.size();
        for (int j = 0; j < sh.nd; ++j) sh.d[j] = dim[tord[j]];
        int perm[kMaxDim];
        for (int j = 0; j < sh.nd; ++j) perm[j] = (int)tord.find(sp.c[j]);
        permute_any(c, Tm, false, sh, perm, C, c32, alpha, beta);
    }
    c.arena.release(mk);
}

void einsum(Ctx& c, const char* spec, double alpha, const T& A, const T& B, double beta, double* C,
            const std::vector<long long>& cdims) {
    einsum_core(c, spec, alpha, A, B, beta, C, false, cdims);
}

void einsum(Ctx& c, const char* spec, double alpha, const T& A, const T& B, double beta, float* C,
            const std::vector<long long>& cdims) {
    einsum_core(c, spec, alpha, A, B, beta, C, true, cdims);
}

}  // namespace adc
