// FP64 subspace kernels of the Davidson iteration; see subspace.cuh.
#include "subspace.cuh"

#include <algorithm>

#include "warp.cuh"

namespace adc {
namespace {

constexpr int kThreads = 256;
constexpr int kRT = 8;  // output rows of a linear combination per pass

// Inner products of a TI x TJ block of (A row, B row) pairs over one slice of x (blockIdx.y), and, in the
// block that finishes a tile last, the sum of its slices' partial results part[tile][slice][TI * TJ] in a
// fixed order.  The block shape follows the problem (TI, TJ <= na, nb rounded up to powers of two), so no
// FP64 FMA is spent on pairs that are not asked for, except in the last tile.  blockIdx.z picks one of two
// pairs of operands.  done: a zero per tile, zero again afterwards.
template <int TI, int TJ>
__global__ void __launch_bounds__(kThreads) k_multidot(int na, const double* __restrict__ A1, const double* __restrict__ A2,
                                                       long long lda, int nb, const double* __restrict__ B1,
                                                       const double* __restrict__ B2, long long ldb, long long n,
                                                       long long chunk, int tiles_j, int trans, double* __restrict__ part,
                                                       unsigned* __restrict__ done, double* __restrict__ D) {
    constexpr int NE = TI * TJ;
    const double *A = blockIdx.z ? A2 : A1, *B = blockIdx.z ? B2 : B1;
    const int ti = blockIdx.x / tiles_j, tj = blockIdx.x % tiles_j;
    const int i0 = ti * TI, j0 = tj * TJ;
    const long long x0 = (long long)blockIdx.y * chunk, x1 = x0 + chunk < n ? x0 + chunk : n;
    double acc[NE];
#pragma unroll
    for (int e = 0; e < NE; ++e) acc[e] = 0.0;
    // rows past na / nb read row 0 (always valid) and are discarded at the end
    const double* Ar[TI];
    const double* Br[TJ];
#pragma unroll
    for (int a = 0; a < TI; ++a) Ar[a] = A + (long long)(i0 + a < na ? i0 + a : 0) * lda;
#pragma unroll
    for (int b = 0; b < TJ; ++b) Br[b] = B + (long long)(j0 + b < nb ? j0 + b : 0) * ldb;
    for (long long x = x0 + threadIdx.x; x < x1; x += kThreads) {
        double bv[TJ];
#pragma unroll
        for (int b = 0; b < TJ; ++b) bv[b] = __ldg(Br[b] + x);
#pragma unroll
        for (int a = 0; a < TI; ++a) {
            const double av = __ldg(Ar[a] + x);
#pragma unroll
            for (int b = 0; b < TJ; ++b) acc[a * TJ + b] = fma(av, bv[b], acc[a * TJ + b]);
        }
    }
    // reduce over the CTA: warp exchange, then one value per warp through shared memory
    __shared__ double red[kThreads];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, e = threadIdx.x % NE;
    warp_fold(acc, lane);
    if (lane % (32 / NE) == 0) red[warp * NE + lane / (32 / NE)] = acc[0];
    __syncthreads();
    double v = 0.0;
    if (threadIdx.x < NE)
        for (int w = 0; w < kThreads / 32; ++w) v += red[w * NE + threadIdx.x];
    if (gridDim.y > 1) {
        const long long tile = (long long)blockIdx.z * gridDim.x + blockIdx.x;
        double* slices = part + tile * gridDim.y * NE;
        if (threadIdx.x < NE) slices[(long long)blockIdx.y * NE + threadIdx.x] = v;
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(done + tile, 1u) == gridDim.y - 1;
        __syncthreads();
        if (!last) return;
        __threadfence();
        double s = 0.0;
        for (int y = threadIdx.x / NE; y < (int)gridDim.y; y += kThreads / NE) s += __ldcg(slices + (long long)y * NE + e);
        red[threadIdx.x] = s;
        for (int w = kThreads / 2; w >= NE; w >>= 1) {
            __syncthreads();
            if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        }
        if (threadIdx.x < NE) v = red[threadIdx.x];
        if (threadIdx.x == 0) done[tile] = 0;
    }
    if (threadIdx.x < NE) {
        const int i = i0 + e / TJ, j = j0 + e % TJ;
        if (i < na && j < nb) D[(long long)blockIdx.z * na * nb + (trans ? (long long)j * na + i : (long long)i * nb + j)] = v;
    }
}

struct DotArgs {
    dim3 grid;
    cudaStream_t st;
    int na, nb;
    const double *A, *A2, *B, *B2;
    long long lda, ldb, n, chunk;
    int tiles_j, trans;
    double* part;
    unsigned* done;
    double* D;
};
template <int TI, int TJ>
void launch_multidot(const DotArgs& q) {
    k_multidot<TI, TJ><<<q.grid, kThreads, 0, q.st>>>(q.na, q.A, q.A2, q.lda, q.nb, q.B, q.B2, q.ldb, q.n, q.chunk, q.tiles_j,
                                                      q.trans, q.part, q.done, q.D);
}

constexpr int kU = 8;  // basis rows loaded ahead of their FMAs (one thread's loads bound a short vector's pass)

// Y[r0 + r][x] = beta Y + alpha sum_i C[(r0 + r) * k + i] V[i][x] for r < NR; C rows in shared memory,
// padded with zeros to kU (the padding reads the last basis row again)
template <int NR>
__global__ void __launch_bounds__(kThreads) k_lincomb(int nr, int k, const double* __restrict__ C,
                                                     const double* __restrict__ V, long long ldv, long long n,
                                                     double alpha, double beta, double* __restrict__ Y, long long ldy) {
    extern __shared__ double Cs[];  // [NR][kp]
    const int kp = (k + kU - 1) / kU * kU;
    for (int e = threadIdx.x; e < NR * kp; e += blockDim.x) Cs[e] = e / kp < nr && e % kp < k ? C[e / kp * k + e % kp] : 0.0;
    __syncthreads();
    for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < n; x += (long long)gridDim.x * blockDim.x) {
        double acc[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) acc[r] = 0.0;
        for (int i0 = 0; i0 < kp; i0 += kU) {
            double v[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) v[u] = __ldg(V + (long long)min(i0 + u, k - 1) * ldv + x);
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (i0 + u < k)
#pragma unroll
                    for (int r = 0; r < NR; ++r) acc[r] = fma(Cs[r * kp + i0 + u], v[u], acc[r]);
        }
#pragma unroll
        for (int r = 0; r < NR; ++r)
            if (r < nr) {
                double* y = Y + (long long)r * ldy + x;
                *y = beta == 0.0 ? alpha * acc[r] : fma(beta, *y, alpha * acc[r]);
            }
    }
}

// the same for two bases: X = C V, R = C W - w X
template <int NR>
__global__ void __launch_bounds__(kThreads) k_ritz(int nr, int k, const double* __restrict__ C, const double* __restrict__ w,
                                                  const double* __restrict__ V, const double* __restrict__ W, long long n,
                                                  double* __restrict__ X, double* __restrict__ R) {
    extern __shared__ double Cs[];  // [NR][kp]
    const int kp = (k + kU - 1) / kU * kU;
    for (int e = threadIdx.x; e < NR * kp; e += blockDim.x) Cs[e] = e / kp < nr && e % kp < k ? C[e / kp * k + e % kp] : 0.0;
    __syncthreads();
    for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < n; x += (long long)gridDim.x * blockDim.x) {
        double a[NR], b[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) a[r] = b[r] = 0.0;
        for (int i0 = 0; i0 < kp; i0 += kU) {
            double v[kU], z[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                v[u] = __ldg(V + (long long)min(i0 + u, k - 1) * n + x);
                z[u] = __ldg(W + (long long)min(i0 + u, k - 1) * n + x);
            }
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (i0 + u < k)
#pragma unroll
                    for (int r = 0; r < NR; ++r) {
                        a[r] = fma(Cs[r * kp + i0 + u], v[u], a[r]);
                        b[r] = fma(Cs[r * kp + i0 + u], z[u], b[r]);
                    }
        }
#pragma unroll
        for (int r = 0; r < NR; ++r)
            if (r < nr) {
                X[(long long)r * n + x] = a[r];
                R[(long long)r * n + x] = fma(-w[r], a[r], b[r]);
            }
    }
}

struct Lower {
    double l[kTriangle * (kTriangle + 1) / 2];  // rows of the lower triangle
};
template <int M>
__global__ void __launch_bounds__(kThreads) k_triangle(int m, Lower L, double* __restrict__ V1, double* __restrict__ V2, long long n) {
    double* V = blockIdx.y ? V2 : V1;
    for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < n; x += (long long)gridDim.x * blockDim.x) {
        double v[M];
#pragma unroll
        for (int j = 0; j < M; ++j) v[j] = j < m ? V[(long long)j * n + x] : 0.0;
#pragma unroll
        for (int r = 0; r < M; ++r)
            if (r < m) {
                double y = 0.0;
#pragma unroll
                for (int j = 0; j <= r; ++j) y = fma(L.l[r * (r + 1) / 2 + j], v[j], y);
                V[(long long)r * n + x] = y;
            }
    }
}

int sm_count() {
    static int n = [] {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return 152;
        return v > 0 ? v : 152;
    }();
    return n;
}

int rows_template(int m) { return m <= 1 ? 1 : m <= 2 ? 2 : m <= 4 ? 4 : 8; }
// short vectors in small blocks, so that they too reach every SM
int block_of(long long n) { return n >= (long long)sm_count() * 4 * kThreads ? kThreads : 64; }
int grid_of(long long n, int threads) { return (int)std::min<long long>((n + threads - 1) / threads, 2048LL / threads * sm_count()); }

}  // namespace

void multidot(Ctx& c, int na, const double* A, long long lda, int nb, const double* B, long long ldb, long long n,
              double* D, const double* A2, const double* B2) {
    if (na <= 0 || nb <= 0) return;
    if (n <= 0) {
        fill(c, (long long)na * nb * (A2 ? 2 : 1), 0.0, D);
        return;
    }
    // the longer side takes the block's TI rows; the result is transposed back if swapped
    const int trans = na < nb ? 1 : 0;
    if (trans) {
        std::swap(na, nb);
        std::swap(A, B);
        std::swap(A2, B2);
        std::swap(lda, ldb);
    }
    const int TI = na >= 8 ? 8 : na > 2 ? 4 : na;          // 1, 2, 4 or 8
    const int TJ = nb >= 4 ? 4 : nb > 2 ? 4 : nb;          // 1, 2 or 4 (TJ <= TI)
    const int ti = (na + TI - 1) / TI, tj = (nb + TJ - 1) / TJ, tiles = ti * tj;
    if ((long long)tiles > (1LL << 30)) throw Error(-1, "multidot: too many vectors");
    // about four resident CTAs per SM in total; each slice at least 512 elements (two per thread: the
    // kernel is bound by the SM's two FP64 FMAs per cycle, so short vectors are spread too)
    long long S = std::max(1LL, (long long)(4 * sm_count()) / tiles);
    S = std::min(S, std::max(1LL, n / 512));
    S = std::min(S, 65535LL);
    const long long chunk = (n + S - 1) / S;
    S = (n + chunk - 1) / chunk;
    const int pairs = A2 ? 2 : 1;
    Arena::Mark mk = c.arena.mark();
    double* part = S > 1 ? c.arena.dalloc((size_t)S * tiles * TI * TJ * pairs) : nullptr;
    unsigned* done = nullptr;  // the context's zeros, or, for more tiles than it has, some of this call's own
    if (S > 1 && tiles * pairs <= Ctx::kDone) {
        done = c.done_counters();
    } else if (S > 1) {
        done = (unsigned*)c.arena.alloc((size_t)tiles * pairs * sizeof(unsigned));
        ADC_CUDA(cudaMemsetAsync(done, 0, (size_t)tiles * pairs * sizeof(unsigned), c.stream));
    }
    const DotArgs q{dim3(tiles, (unsigned)S, pairs), c.stream, na, nb, A, A2, B, B2, lda, ldb, n, chunk, tj, trans, part, done, D};
    switch (TI * 16 + TJ) {
        case 8 * 16 + 4: launch_multidot<8, 4>(q); break;
        case 8 * 16 + 2: launch_multidot<8, 2>(q); break;
        case 8 * 16 + 1: launch_multidot<8, 1>(q); break;
        case 4 * 16 + 4: launch_multidot<4, 4>(q); break;
        case 4 * 16 + 2: launch_multidot<4, 2>(q); break;
        case 4 * 16 + 1: launch_multidot<4, 1>(q); break;
        case 2 * 16 + 2: launch_multidot<2, 2>(q); break;
        case 2 * 16 + 1: launch_multidot<2, 1>(q); break;
        case 1 * 16 + 1: launch_multidot<1, 1>(q); break;
        default: throw Error(-1, "multidot: no block shape");
    }
    ++c.kernels;
    ADC_CUDA(cudaGetLastError());
    c.arena.release(mk);
}

void lincomb(Ctx& c, int nr, int k, const double* C, const double* V, long long ldv, long long n, double alpha, double beta,
             double* Y, long long ldy) {
    if (nr <= 0 || n <= 0) return;
    if (k <= 0) {
        for (int r = 0; r < nr; ++r) {
            double* y = Y + (long long)r * ldy;
            if (beta == 0.0)
                fill(c, n, 0.0, y);
            else
                axpby(c, n, beta, y, 0.0, y);
        }
        return;
    }
    const long long kp = (k + kU - 1) / kU * kU;
    if (kRT * kp * sizeof(double) > 48 * 1024) throw Error(-1, "lincomb: basis too large (k > 768)");
    for (int r0 = 0; r0 < nr; r0 += kRT) {
        const int m = std::min(kRT, nr - r0);
        const int NR = rows_template(m), threads = block_of(n);
        const int grid = grid_of(n, threads);
        const double* Cr = C + (long long)r0 * k;
        double* Yr = Y + (long long)r0 * ldy;
        const size_t smem = (size_t)NR * kp * sizeof(double);
        switch (NR) {
            case 1: k_lincomb<1><<<grid, threads, smem, c.stream>>>(m, k, Cr, V, ldv, n, alpha, beta, Yr, ldy); break;
            case 2: k_lincomb<2><<<grid, threads, smem, c.stream>>>(m, k, Cr, V, ldv, n, alpha, beta, Yr, ldy); break;
            case 4: k_lincomb<4><<<grid, threads, smem, c.stream>>>(m, k, Cr, V, ldv, n, alpha, beta, Yr, ldy); break;
            default: k_lincomb<8><<<grid, threads, smem, c.stream>>>(m, k, Cr, V, ldv, n, alpha, beta, Yr, ldy);
        }
        ++c.kernels;
        ADC_CUDA(cudaGetLastError());
    }
}

void ritz(Ctx& c, int nr, int k, const double* C, const double* w, const double* V, const double* W, long long n, double* X,
          double* R) {
    const long long kp = (k + kU - 1) / kU * kU;
    if (k <= 0 || kRT * kp * sizeof(double) > 48 * 1024) throw Error(-1, "lincomb: basis too large (k > 768)");
    for (int r0 = 0; r0 < nr; r0 += kRT) {
        const int m = std::min(kRT, nr - r0), NR = rows_template(m), threads = block_of(n), grid = grid_of(n, threads);
        const double* Cr = C + (long long)r0 * k;
        double *Xr = X + r0 * n, *Rr = R + r0 * n;
        const size_t smem = (size_t)NR * kp * sizeof(double);
        switch (NR) {
            case 1: k_ritz<1><<<grid, threads, smem, c.stream>>>(m, k, Cr, w + r0, V, W, n, Xr, Rr); break;
            case 2: k_ritz<2><<<grid, threads, smem, c.stream>>>(m, k, Cr, w + r0, V, W, n, Xr, Rr); break;
            case 4: k_ritz<4><<<grid, threads, smem, c.stream>>>(m, k, Cr, w + r0, V, W, n, Xr, Rr); break;
            default: k_ritz<8><<<grid, threads, smem, c.stream>>>(m, k, Cr, w + r0, V, W, n, Xr, Rr);
        }
        ++c.kernels;
        ADC_CUDA(cudaGetLastError());
    }
}

void triangle(Ctx& c, int m, const double* L, double* V, double* V2, long long n) {
    if (m <= 0 || n <= 0) return;
    if (m > kTriangle) throw Error(-1, "triangle: too many vectors");
    Lower q{};
    for (int r = 0; r < m; ++r)
        for (int j = 0; j <= r; ++j) q.l[r * (r + 1) / 2 + j] = L[r * m + j];
    const int threads = block_of(n);
    const dim3 grid(grid_of(n, threads), 2);
    if (m <= 4)
        k_triangle<4><<<grid, threads, 0, c.stream>>>(m, q, V, V2, n);
    else
        k_triangle<kTriangle><<<grid, threads, 0, c.stream>>>(m, q, V, V2, n);
    ++c.kernels;
    ADC_CUDA(cudaGetLastError());
}

}  // namespace adc
