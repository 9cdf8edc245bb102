// FP64-accurate contractions on the BF16 tensor cores of sm_103a.
//
// GB300 has about 1.2 TFLOP/s of FP64 against 2 PFLOP/s of dense BF16, so an FP64 product is
// cheaper as a sum of exact integer products (the error-free splitting of Ozaki, Ogita, Oishi and
// Rump, Numer. Algorithms 59, 95 (2012)):
//   * every row of A and of B is scaled by a power of two to integers below 2^63 in size and cut
//     into eight signed digits of eight bits (|d| <= 128), which BF16 holds exactly;
//   * the digit products of equal weight, s = i + j, accumulate in one FP32 tensor-memory
//     accumulator per s.  Over 128 summed terms and at most eight digit pairs such a sum stays within
//     8 * 128 * 2^14 = 2^24, so it is an exact integer; then it is drained into 64-bit integer
//     registers, where it stays exact over a slice of up to 2^23 terms (longer K is cut into slices);
//   * the weights s = 14 .. 7 are kept (36 of 64 digit pairs).  What is left out of a sum of K terms is at most
//     2^-61 K of the product of the row scales (seven pairs of weight 6 to a term, all of one sign at their
//     largest: constant rows), and for digits of random signs about 2^-63 sqrt(K).  The one rounding of the
//     result is to FP64.  (Seven digits and 34 pairs round the inputs to 2^-57 of their rows' largest element,
//     which an integral row with a coherent diagonal, (ia|ia) 20 times the others, turns into 1.2e-16 of the
//     result.)
// So a product is fixed point to 63 bits of its rows' largest elements: in norm as accurate as an FP64 GEMM,
// but an element 2^-63 below its row's largest does not count, where floating point would keep it.  A row
// with an infinity or a NaN gives NaN.
// Norm of the error over norm of an FP64 sigma of 5 vectors, against long double: 7.4e-17 (IP 8/48/180) and
// 7.9e-17 (EA 6/40/150), with DGEMM 1.5e-16 and 5.9e-16.
// Measured, the IP sigma of 5 vectors at 14/113/445: 24.6 -> 3.8 ms in 20 contractions, 0.30 ms with the coupling block held
// (three of 70 x 1582 x 1582 results and terms take 37 us each: 40 MB of cached digits read from L2 by 99
// tiles; other tile widths, slices and the exchanged sides are all between 34 and 140 us); the FP64 setup of
// an IP molecule at 17/121/483 with its first sigma 217 -> 18.7 ms, about half of it here (23.2 ms with the mapping
// of its memory, where no other handle lives: memory.cuh).
//
// Tile: 128 rows of A x BNT columns (16 .. 64) of B per CTA, because the eight accumulators take
// 8 x BNT of the 512 tensor-memory columns.  The digit planes of B lie one after another in shared
// memory as further rows of one K-major operand and the accumulators of consecutive weights are
// consecutive in tensor memory, so that one MMA multiplies digit i of A with up to 256 / BNT digits
// of B: 12 MMAs of up to 256 columns per 16-deep K step instead of 36 of 64 (which would be bound by
// reading A from shared memory 36 times).
#include <cooperative_groups.h>

#include <algorithm>
#include <cstdint>
#include <mutex>

#include "digits.cuh"
#include "gemm64.cuh"
#include "plan64.cuh"
#include "tcgen05.cuh"

namespace adc {

namespace {

constexpr int G_EPI = 8;       // epilogue warps
constexpr int G_THREADS = 64 + 32 * G_EPI;
constexpr int G_MAXST = 4;
constexpr size_t G_SMEM = 226 * 1024;

// ---- digits -------------------------------------------------------------------------
constexpr int DT = 256;  // threads of the digit kernels
constexpr int DR = 8;    // rows per block at most

struct DigitSide {
    Operand64 x;
    long long Kp;
    __nv_bfloat16* out;  // [ND] planes, `plane` apart, of [rows][Kp]; digit 0 the least significant
    long long plane;
    int* ex;             // biased exponent field of the row's largest element (0x7ff: not finite)
    int row_lanes;       // the tensor's contiguous axis is the last row axis (else the lanes run along k)
    int R;               // rows per block, a power of two
};

__device__ __forceinline__ double ld_op(const Operand64& x, long long i) {
    return x.f32 ? (double)((const float*)x.p)[i] : ((const double*)x.p)[i];
}

__device__ __forceinline__ long long digit_row(const Operand64& x, unsigned r) {
    long long off = 0;
    for (int j = x.nr - 1; j >= 0; --j) {
        const unsigned d = (unsigned)x.rd[j], q = r / d;
        off += (long long)(r - q * d) * x.rs[j];
        r = q;
    }
    return off;
}
__device__ __forceinline__ long long digit_k(const Operand64& x, unsigned k) {
    long long off = 0;
    for (int j = x.nk - 1; j >= 0; --j) {
        const unsigned d = (unsigned)x.kd[j], q = k / d;
        off += (long long)(k - q * d) * x.ks[j];
        k = q;
    }
    return off;
}
// x[0], x[1] of a row of largest exponent field ef -> their digits, at `at` of each plane
__device__ __forceinline__ void put_digits(const DigitSide& sd, long long at, const double* x, int ef) {
    unsigned dig[ND];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const long long v = scaled_integer((uint64_t)__double_as_longlong(x[h]), ef);
        const uint64_t w = with_carries(v);
#pragma unroll
        for (int p = 0; p < ND; ++p) {
            // a small integer's BF16 bits are the upper half of its FP32 bits
            const unsigned u = __float_as_uint((float)digit(v, w, p)) >> 16;
            dig[p] = h == 0 ? u : dig[p] | (u << 16);
        }
    }
#pragma unroll
    for (int p = 0; p < ND; ++p) *(unsigned*)(sd.out + p * sd.plane + at) = dig[p];
}

// Rows of up to 8 DSEG terms: both operands in one launch (blocks [0, blocks_a) of x the rows of A), a
// row's K over the blocks of a cluster, seg terms each in shared memory.  The rows' largest exponents go
// around through distributed shared memory, so every element is read once and neither a second launch
// nor a cleared array is needed (70 rows of 1582: 5.8 us, against 8.5 + 9.7 and 1.1 for the clearing).
constexpr int DSEG = 512;
__global__ void __launch_bounds__(DT) k_digits(const __grid_constant__ DigitSide sa, const __grid_constant__ DigitSide sb,
                                               int blocks_a, int seg) {
    extern __shared__ double tile[];  // [R][seg + 1]
    __shared__ long long offk[DSEG], offr[DR];
    __shared__ int emax[DR], eall[DR];
    const bool isb = (int)blockIdx.x >= blocks_a;
    const DigitSide& sd = isb ? sb : sa;
    const Operand64& x = sd.x;
    const int R = sd.R, tid = threadIdx.x, ld = seg + 1;
    const long long row0 = (long long)(isb ? blockIdx.x - blocks_a : blockIdx.x) * R, k0 = (long long)blockIdx.y * seg;
    if (tid < R) {
        offr[tid] = digit_row(x, (unsigned)min(row0 + tid, x.rows - 1));
        emax[tid] = 0;
    }
    for (int k = tid; k < seg; k += DT) offk[k] = digit_k(x, (unsigned)min(k0 + k, x.K - 1));
    __syncthreads();
    const int per = DT / R, lper = 31 - __clz(per), lR = 8 - lper;
    if (sd.row_lanes) {
        const int rr = tid & (R - 1);
#pragma unroll 4
        for (int k = tid >> lR; k < seg; k += per)
            tile[rr * ld + k] = k0 + k < x.K && row0 + rr < x.rows ? ld_op(x, offr[rr] + offk[k]) : 0.0;
    } else {
        for (int rr = 0; rr < R; ++rr)
#pragma unroll
            for (int k = tid; k < seg; k += DT)
                tile[rr * ld + k] = k0 + k < x.K && row0 + rr < x.rows ? ld_op(x, offr[rr] + offk[k]) : 0.0;
    }
    __syncthreads();
    const int r = tid >> lper, t = tid & (per - 1);  // per threads to a row
    int m = 0;
    for (int k = t; k < seg; k += per) m = max(m, exponent_of((uint64_t)__double_as_longlong(tile[r * ld + k])));
    if (m > 0) atomicMax(&emax[r], m);
    namespace cg = cooperative_groups;
    const cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    if (tid < R) {
        int e = 0;
        for (unsigned q = 0; q < cl.num_blocks(); ++q) e = max(e, *cl.map_shared_rank(&emax[tid], q));
        eall[tid] = e;
        if (blockIdx.y == 0 && row0 + tid < x.rows) sd.ex[row0 + tid] = e;
    }
    cl.sync();  // (no block leaves while its maxima are read)
    if (row0 + r >= x.rows) return;
    const int ef = eall[r];
    for (int k = 2 * t; k < seg && k0 + k < sd.Kp; k += 2 * per) put_digits(sd, (row0 + r) * sd.Kp + k0 + k, tile + r * ld + k, ef);
}

// Longer rows: K in segments of kseg along y and two launches, pass 1 the rows' largest exponents (into
// ex, zero before), pass 2 the digits.
__global__ void __launch_bounds__(DT) k_digits_long(const __grid_constant__ DigitSide sa, const __grid_constant__ DigitSide sb,
                                                    int blocks_a, long long kseg, int pass) {
    __shared__ double tile[DR][DT + 1];
    __shared__ long long offk[DT], offr[DR];
    __shared__ int emax[DR];
    const bool isb = (int)blockIdx.x >= blocks_a;
    const DigitSide& sd = isb ? sb : sa;
    const Operand64& x = sd.x;
    const int R = sd.R, tid = threadIdx.x;
    const long long row0 = (long long)(isb ? blockIdx.x - blocks_a : blockIdx.x) * R;
    const long long kbeg = blockIdx.y * kseg, kend = min(sd.Kp, kbeg + kseg);
    if (tid < R) {
        offr[tid] = digit_row(x, (unsigned)min(row0 + tid, x.rows - 1));
        emax[tid] = pass == 2 ? sd.ex[min(row0 + tid, x.rows - 1)] : 0;
    }
    const int per = DT / R, lper = 31 - __clz(per), lR = 8 - lper;  // threads per row when the lanes run along k
    const int r = tid >> lper;
    for (long long k0 = kbeg; k0 < kend; k0 += DT) {
        __syncthreads();
        offk[tid] = digit_k(x, (unsigned)min(k0 + tid, x.K - 1));
        __syncthreads();
        for (int e = tid; e < R * DT; e += DT) {
            const int rr = sd.row_lanes ? e & (R - 1) : e >> 8, k = sd.row_lanes ? e >> lR : e & (DT - 1);
            tile[rr][k] = k0 + k < x.K && row0 + rr < x.rows ? ld_op(x, offr[rr] + offk[k]) : 0.0;
        }
        __syncthreads();
        if (pass == 1) {
            int m = 0;
            for (int k = tid & (per - 1); k < DT; k += per) m = max(m, exponent_of((uint64_t)__double_as_longlong(tile[r][k])));
            if (m > 0) atomicMax(&emax[r], m);
        } else if (row0 + r < x.rows) {
            for (int k = 2 * (tid & (per - 1)); k < DT && k0 + k < sd.Kp; k += 2 * per)
                put_digits(sd, (row0 + r) * sd.Kp + k0 + k, &tile[r][k], emax[r]);
        }
    }
    __syncthreads();
    if (pass == 1 && tid < R && row0 + tid < x.rows) atomicMax(&sd.ex[row0 + tid], emax[tid]);
}

// ---- GEMM ---------------------------------------------------------------------------
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* m, uint64_t* bar, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(
            su32(dst)),
        "l"((uint64_t)m), "r"(su32(bar)), "r"(x), "r"(y), "r"(0)
        : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}
// K-major descriptor of 64-byte rows in the 64-byte swizzle (8-row groups of 512 bytes)
__device__ __forceinline__ uint64_t desc64(const void* p) {
    return (uint64_t)((su32(p) >> 4) & 0x3FFF) | (uint64_t)1 << 16 | (uint64_t)(512 >> 4) << 32 | (uint64_t)1 << 46 |
           (uint64_t)4 << 61;
}

struct Gemm64Out {
    int M, N, mt, nt, S, slice_kb;  // slices of slice_kb K blocks
    const int *ea, *eb;
    double* T;  // [S][M][N], or NULL: o
    Out64 o;
    int* err;
};

__device__ __forceinline__ long long axes_offset(int n, const long long* d, const long long* st, unsigned x) {
    long long off = 0;
    for (int j = n - 1; j >= 0; --j) {
        const unsigned dj = (unsigned)d[j], q = x / dj;
        off += (long long)(x - q * dj) * st[j];
        x = q;
    }
    return off;
}
// out = alpha v + beta out
__device__ __forceinline__ void put64(const Out64& o, long long at, double v) {
    if (o.alpha != 1.0) v *= o.alpha;
    if (o.beta != 0.0) v += o.beta == 1.0 ? o.p[at] : o.beta * o.p[at];
    o.p[at] = v;
}

// The digit products of one 16-deep K step: every MMA multiplies digit i of A with nj digits of B.
// Unrolled at compile time: one thread issues them all, and address arithmetic between them would
// cost it more than the MMAs take.  kFirst: first step of an epoch (accumulators are started).
template <int BNT, bool kFirst>
__device__ __forceinline__ void digit_products(uint32_t tmem, uint64_t a, uint64_t b) {
    constexpr uint32_t ib = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(GM >> 4) << 24);
    constexpr int jmax = 256 / BNT;  // digits of B per MMA
#pragma unroll
    for (int i = ND - 1; i >= 0; --i) {
        const int j = SMIN - i;  // (the top digit of A meets every digit of B and starts all accumulators)
        const int parts = (ND - j + jmax - 1) / jmax, nj = (ND - j + parts - 1) / parts;  // nearly equal widths
#pragma unroll
        for (int q = 0; q < parts; ++q) {
            const int j0 = j + q * nj, n = nj < ND - j0 ? nj : ND - j0;
            mma_bf16(tmem + (uint32_t)((i + j0 - SMIN) * BNT), a + (uint64_t)(i * (GM * GK * 2 >> 4)),
                     b + (uint64_t)(j0 * (BNT * GK * 2 >> 4)), ib | ((uint32_t)(n * BNT >> 3) << 17),
                     kFirst && i == ND - 1 ? 0u : 1u);
        }
    }
}

template <int BNT>
__global__ void __launch_bounds__(G_THREADS, 1)
    k_gemm64(const __grid_constant__ CUtensorMap ma, const __grid_constant__ CUtensorMap mb, int num_k, int stages,
             const __grid_constant__ Gemm64Out o) {
    constexpr int tmem_cols = BNT <= 16 ? 128 : BNT <= 32 ? 256 : 512;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ uint64_t full_bar[G_MAXST], empty_bar[G_MAXST], tfull, tempty, done_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int A_PL = GM * GK * 2, B_PL = BNT * GK * 2;
    constexpr int STAGE = ND * (A_PL + B_PL);
    const int tiles = o.mt * o.nt, nunits = tiles * o.S;
    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        mbar_init(&tfull, 1);
        mbar_init(&tempty, G_EPI);
        mbar_init(&done_bar, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&tmem_slot)), "r"(tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            long long g = 0;
            for (int u = blockIdx.x; u < nunits && !abort_flag; u += gridDim.x) {
                const int sl = u / tiles, t = u - sl * tiles, m_tile = t % o.mt, n_tile = t / o.mt;
                const int kb1 = min(num_k, (sl + 1) * o.slice_kb);
                for (int kb = sl * o.slice_kb; kb < kb1; ++kb, ++g) {
                    const int s = (int)(g % stages);
                    if (g >= stages && !mbar_wait(&empty_bar[s], (uint32_t)(((g / stages) & 1) ^ 1), &abort_flag, o.err)) break;
                    uint8_t* st = smem + (size_t)s * STAGE;
                    mbar_expect_tx(&full_bar[s], STAGE);
                    tma_load_3d(st, &ma, &full_bar[s], kb * GK, m_tile * GM);
                    tma_load_3d(st + ND * A_PL, &mb, &full_bar[s], kb * GK, n_tile * BNT);
                }
            }
            if (abort_flag) {
                // let the copies of the last `stages` issues land before the CTA retires (bounded)
                for (long long q = (g > stages ? g - stages : 0); q < g; ++q) {
                    const uint64_t t0 = gtime();
                    while (!mbar_try(&full_bar[q % stages], (uint32_t)((q / stages) & 1)) && gtime() - t0 < WAIT_NS) {
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            long long g = 0, e = 0;
            bool ok = true;
            for (int u = blockIdx.x; u < nunits && ok && !abort_flag; u += gridDim.x) {
                const int sl = u / tiles, kb0 = sl * o.slice_kb, kb1 = min(num_k, kb0 + o.slice_kb);
                for (int kb = kb0; kb < kb1; ++kb, ++g) {
                    const int s = (int)(g % stages), in_epoch = (kb - kb0) % EPOCH;
                    if (!mbar_wait(&full_bar[s], (uint32_t)((g / stages) & 1), &abort_flag, o.err) ||
                        (in_epoch == 0 && e > 0 && !mbar_wait(&tempty, (uint32_t)((e & 1) ^ 1), &abort_flag, o.err))) {
                        ok = false;
                        break;
                    }
                    fence_after();
                    const uint64_t a0 = desc64(smem + (size_t)s * STAGE), b0 = desc64(smem + (size_t)s * STAGE + ND * A_PL);
                    if (in_epoch == 0)
                        digit_products<BNT, true>(tmem, a0, b0);
                    else
                        digit_products<BNT, false>(tmem, a0, b0);
                    digit_products<BNT, false>(tmem, a0 + 2, b0 + 2);  // 16 BF16 = 32 bytes along K
                    mma_commit(&empty_bar[s]);
                    if (in_epoch == EPOCH - 1 || kb == kb1 - 1) {
                        mma_commit(&tfull);
                        ++e;
                    }
                }
            }
            mma_commit(&done_bar);
        }
    } else {
        const int ew = warp - 2, quarter = warp & 3, half = ew >> 2;
        constexpr int cw = BNT / 2;
        const int cbeg = half * cw;
        // staging of the results (after the pipeline stages): a row of 8 results per lane, padded
        double* stg = (double*)(smem + (size_t)stages * STAGE) + ew * 32 * 9;
        long long e = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < nunits && ok; u += gridDim.x) {
            const int sl = u / tiles, t = u - sl * tiles, m_tile = t % o.mt, n_tile = t / o.mt;
            const int kb0 = sl * o.slice_kb, epochs = (min(num_k, kb0 + o.slice_kb) - kb0 + EPOCH - 1) / EPOCH;
            long long hi[cw], lo[cw];
#pragma unroll
            for (int q = 0; q < cw; ++q) hi[q] = lo[q] = 0;
            for (int i = 0; i < epochs; ++i, ++e) {
                if (!mbar_wait(&tfull, (uint32_t)(e & 1), &abort_flag, o.err)) {
                    ok = false;
                    break;
                }
                fence_after();
                const uint32_t base = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)cbeg;
#pragma unroll
                for (int c0 = 0; c0 < cw; c0 += 8) {
                    uint32_t r[NL][8];
#pragma unroll
                    for (int l = 0; l < NL; ++l) tmem_ld8(base + (uint32_t)(l * BNT + c0), r[l]);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        int v[NL];
#pragma unroll
                        for (int l = 0; l < NL; ++l) v[l] = __float2int_rn(__uint_as_float(r[l][q]));
                        hi[c0 + q] += (long long)v[7] * (1 << 24) + (long long)v[6] * (1 << 16) + (long long)v[5] * (1 << 8) + v[4];
                        lo[c0 + q] += (long long)v[3] * (1 << 24) + (long long)v[2] * (1 << 16) + (long long)v[1] * (1 << 8) + v[0];
                    }
                }
                fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&tempty);
            }
            if (!ok) break;
            const int row0 = m_tile * GM + quarter * 32, row = row0 + lane, colt = n_tile * BNT + cbeg;
            if (row0 >= o.M || colt >= o.N) continue;  // uniform over the warp
            const int ea = row < o.M ? o.ea[row] : 0;
            const long long orow = o.T ? ((long long)sl * o.M + row) * o.N : axes_offset(o.o.nr, o.o.rd, o.o.rs, (unsigned)row);
#pragma unroll
            for (int c0 = 0; c0 < cw; c0 += 8) {
                // 32 rows x 8 columns through shared memory: whole sectors of the output rows
                const int ebl = colt + c0 + (lane & 7) < o.N ? o.eb[colt + c0 + (lane & 7)] : 0;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int eb = __shfl_sync(0xffffffffu, ebl, q);
                    // weights: digit products of weight s carry 2^(8 s); hi starts at s = 11, lo at s = 7;
                    // a row's integers carry 2^(ef - 1085)
                    stg[lane * 9 + q] = ea == 0x7ff || eb == 0x7ff ? __longlong_as_double(0x7ff8000000000000LL)
                                                                  : to_double(hi[c0 + q], lo[c0 + q], 8 * SMIN + ea + eb - 2 * 1085);
                }
                __syncwarp();
                const int col = colt + c0 + (lane & 7);
                const long long ocol = o.T ? col : axes_offset(o.o.nc, o.o.cd, o.o.cs, (unsigned)col);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int rr = i * 4 + (lane >> 3);
                    const long long at = __shfl_sync(0xffffffffu, orow, rr) + ocol;
                    if (row0 + rr < o.M && col < o.N) {
                        if (o.T)
                            o.T[at] = stg[rr * 9 + (lane & 7)];
                        else
                            put64(o.o, at, stg[rr * 9 + (lane & 7)]);
                    }
                }
                __syncwarp();
            }
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 1) {
        const uint64_t t0 = gtime();
        while (!mbar_try(&done_bar, 0) && gtime() - t0 < WAIT_NS) {
        }
        fence_after();
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");
    }
}

// digit planes as a 3-D tensor {k, row, digit}, box {GK, box_rows, ND}, 64-byte swizzle
CUtensorMap make_map_digits(const Digits64& d, int box_rows) {
    const long long rows = d.rows, Kp = d.Kp;
    CUtensorMap m;
    cuuint64_t dims[3] = {(cuuint64_t)Kp, (cuuint64_t)rows, ND};
    cuuint64_t strides[2] = {(cuuint64_t)Kp * 2, (cuuint64_t)(d.plane * 2)};
    cuuint32_t box[3] = {GK, (cuuint32_t)box_rows, ND};
    cuuint32_t es[3] = {1, 1, 1};
    const CUresult r = tensor_map_encoder()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, d.d, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) throw Error(-3, "cuTensorMapEncodeTiled (digits) failed: " + std::to_string((int)r));
    return m;
}

int sm_count() {
    int dev = 0, n = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n;
}

void launch64(Ctx& c, const Digits64& A, const Digits64& B, const Gemm64Plan& p, double* T, const Out64& out) {
    if (!c.d_err) {
        if (c.capturing) throw Error(-3, "error flag allocation during stream capture");
        c.d_err = (int*)dev_alloc(sizeof(int), c.stream);
        ADC_CUDA(cudaMemsetAsync(c.d_err, 0, sizeof(int), c.stream));
    }
    const int sms = sm_count(), num_k = (int)((A.Kp + GK - 1) / GK);
    const CUtensorMap ma = make_map_digits(A, GM), mb = make_map_digits(B, p.BNT);
    Gemm64Out o{};
    o.M = (int)A.rows;
    o.N = (int)B.rows;
    o.mt = (int)((A.rows + GM - 1) / GM);
    o.nt = (int)((B.rows + p.BNT - 1) / p.BNT);
    o.S = p.S;
    o.slice_kb = p.kb;
    o.ea = A.ex;
    o.eb = B.ex;
    o.T = T;
    o.o = out;
    o.err = c.d_err;
    const long long units = (long long)o.mt * o.nt * p.S;
    if (units > (1LL << 30)) throw Error(-1, "gemm64: too many tiles");
    const int stage = ND * (GM + p.BNT) * GK * 2;
    const int stages = std::min(G_MAXST, (int)((G_SMEM - 1024 - G_EPI * 32 * 9 * sizeof(double)) / stage));
    static std::once_flag once[64];
    int dev = 0;
    ADC_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) throw Error(-3, "gemm64: device index out of range");
    std::call_once(once[dev], [] {
        for (auto k : {k_gemm64<16>, k_gemm64<32>, k_gemm64<48>, k_gemm64<64>})
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G_SMEM);
    });
    const auto kern = p.BNT == 16 ? k_gemm64<16> : p.BNT == 32 ? k_gemm64<32> : p.BNT == 48 ? k_gemm64<48> : k_gemm64<64>;
    kern<<<(unsigned)std::min<long long>(units, sms), G_THREADS, G_SMEM, c.stream>>>(ma, mb, num_k, stages, o);
    ++c.kernels;
    ADC_CUDA(cudaGetLastError());
}

}  // namespace

bool gemm64_fits(long long M, long long N, long long K) {
    return M < (1LL << 30) && N < (1LL << 30) && K < (1LL << 30) && 2.0 * M * N * K >= 4e6;
}

size_t digits64_bytes(long long rows, long long K) {
    return (size_t)ND * rows * ((K + 7) / 8 * 8) * 2 + ((size_t)rows * sizeof(int) + 255) / 256 * 256;
}
Digits64 digits64_in(void* buffer, long long rows, long long K) {
    Digits64 d;
    d.rows = rows;
    d.Kp = (K + 7) / 8 * 8;
    d.plane = rows * d.Kp;
    d.d = (__nv_bfloat16*)buffer;
    d.ex = (int*)(d.d + ND * d.plane);
    return d;
}

void digitise64(Ctx& c, const Operand64* x, Digits64* out, int n) {
    DigitSide side[2];
    int blocks[2] = {0, 0};
    const int sms = sm_count();
    const long long Kp = out[0].Kp;
    // one launch where a cluster's eight blocks hold a row: as few blocks to a row as hold it, more (of at
    // least 256 terms) while the launch leaves SMs idle
    const bool once = Kp <= 8 * DSEG;
    long long rows8 = 0;
    for (int i = 0; i < n; ++i) rows8 += (x[i].rows + DR - 1) / DR;
    long long cs = std::max<long long>(1, (Kp + DSEG - 1) / DSEG);
    while (once && cs < 8 && Kp > 256 * cs && rows8 * cs < 2 * sms) ++cs;
    const long long seg = once ? ((Kp + cs - 1) / cs + 255) / 256 * 256 : DSEG;
    cs = (Kp + seg - 1) / seg;
    for (int i = 0; i < n; ++i) {
        DigitSide& d = side[i];
        d.x = x[i];
        d.Kp = Kp;
        d.out = out[i].d;
        d.plane = out[i].plane;
        d.ex = out[i].ex;
        if (x[i].K > Kp || out[i].Kp != Kp) throw Error(-1, "digitise64: shape mismatch");
        long long smallest = d.x.nk > 0 ? d.x.ks[d.x.nk - 1] : 1;
        d.row_lanes = 0;
        for (int j = 0; j < d.x.nk; ++j) smallest = std::min(smallest, d.x.kd[j] > 1 ? d.x.ks[j] : smallest);
        for (int j = 0; j < d.x.nr; ++j)
            if (d.x.rd[j] > 1 && d.x.rs[j] < smallest) d.row_lanes = 1;
        d.R = DR;
        while (d.R > 1 && (d.x.rows + d.R - 1) / d.R * cs < 2 * sms) d.R /= 2;
        const long long nb = (d.x.rows + d.R - 1) / d.R;
        if (nb > (1LL << 30)) throw Error(-1, "gemm64: too many rows");
        blocks[i] = (int)nb;
    }
    if (n < 2) side[1] = side[0];
    const unsigned bx = (unsigned)(blocks[0] + blocks[1]);
    if (once) {
        const int R = std::max(side[0].R, side[1].R);
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute cl[1];
        cl[0].id = cudaLaunchAttributeClusterDimension;
        cl[0].val.clusterDim.x = 1;
        cl[0].val.clusterDim.y = (unsigned)cs;
        cl[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(bx, (unsigned)cs);
        cfg.blockDim = dim3(DT);
        cfg.dynamicSmemBytes = (size_t)R * (seg + 1) * sizeof(double);
        cfg.stream = c.stream;
        cfg.attrs = cl;
        cfg.numAttrs = 1;
        ADC_CUDA(cudaLaunchKernelEx(&cfg, k_digits, side[0], side[1], blocks[0], (int)seg));
        ++c.kernels;
    } else {
        for (int i = 0; i < n; ++i)
            ADC_CUDA(cudaMemsetAsync(side[i].ex, 0, (size_t)side[i].x.rows * sizeof(int), c.stream));
        for (int pass = 1; pass <= 2; ++pass) {
            long long ks = seg;
            while ((Kp + ks - 1) / ks > 65535) ks *= 2;
            k_digits_long<<<dim3(bx, (unsigned)((Kp + ks - 1) / ks)), DT, 0, c.stream>>>(side[0], side[1], blocks[0], ks, pass);
            ++c.kernels;
        }
    }
    ADC_CUDA(cudaGetLastError());
}

double* gemm64(Ctx& c, const Operand64& A, const Digits64* da, const Operand64& B, const Digits64* db, const Out64& out,
               int& S) {
    const long long M = da ? da->rows : A.rows, N = db ? db->rows : B.rows, Kp = da ? da->Kp : (A.K + 7) / 8 * 8;
    const Gemm64Plan plan = plan64(M, N, Kp, sm_count());
    S = plan.S;
    // (the result is allocated first: it outlives the digits)
    double* T = out.p && S == 1 ? nullptr : c.arena.dalloc((size_t)S * M * N);
    Arena::Mark mk = c.arena.mark();
    Digits64 d[2], todo[2];
    Operand64 x[2];
    int n = 0;
    for (int i = 0; i < 2; ++i) {
        const Digits64* have = i ? db : da;
        const Operand64& op = i ? B : A;
        d[i] = have ? *have : digits64_in(c.arena.alloc(digits64_bytes(op.rows, op.K)), op.rows, op.K);
        if (!have) x[n] = op, todo[n++] = d[i];
    }
    if (n) digitise64(c, x, todo, n);
    launch64(c, d[0], d[1], plan, T, out);
    c.arena.release(mk);
    return T;
}

// ---- the smallest contractions, in FP64 arithmetic ---------------------------------------------
// 8 x 8 outputs per block of 64 threads: at two FP64 FMAs per cycle and SM, work of this size is only
// quick when it is spread over all SMs.  Operands and output are reached through their strides, so a
// contraction is one launch (with K slices: and the permute that sums them).
namespace {
constexpr int ST = 8, SK = 32;

__global__ void __launch_bounds__(ST * ST) k_small64(const __grid_constant__ Operand64 A, const __grid_constant__ Operand64 B,
                                                     long long kslice, double* __restrict__ T, const __grid_constant__ Out64 o) {
    __shared__ double as[ST][SK + 1], bs[ST][SK + 1];
    __shared__ long long ra[ST], rb[ST], ka[SK], kb[SK];
    const int t = threadIdx.x, ti = t / ST, tj = t % ST;
    const long long m0 = blockIdx.y * (long long)ST, n0 = blockIdx.x * (long long)ST;
    if (t < ST) ra[t] = axes_offset(A.nr, A.rd, A.rs, (unsigned)min(m0 + t, A.rows - 1));
    if (t >= 32 && t < 32 + ST) rb[t - 32] = axes_offset(B.nr, B.rd, B.rs, (unsigned)min(n0 + t - 32, B.rows - 1));
    const long long k0 = blockIdx.z * kslice, k1 = min(A.K, k0 + kslice);
    double acc = 0.0;
    for (long long kc = k0; kc < k1; kc += SK) {
        __syncthreads();
        const unsigned k = (unsigned)min(kc + (t & 31), A.K - 1);
        if (t < 32)
            ka[t] = axes_offset(A.nk, A.kd, A.ks, k);
        else
            kb[t - 32] = axes_offset(B.nk, B.kd, B.ks, k);
        __syncthreads();
#pragma unroll
        for (int e = t; e < ST * SK; e += ST * ST) {
            const int r = e / SK, q = e % SK;
            as[r][q] = kc + q < k1 ? ld_op(A, ra[r] + ka[q]) : 0.0;
            bs[r][q] = kc + q < k1 ? ld_op(B, rb[r] + kb[q]) : 0.0;
        }
        __syncthreads();
        const int kn = (int)min((long long)SK, k1 - kc);
        for (int q = 0; q < kn; ++q) acc = fma(as[ti][q], bs[tj][q], acc);
    }
    const long long m = m0 + ti, n = n0 + tj;
    if (m < A.rows && n < B.rows) {
        if (T)
            T[(blockIdx.z * A.rows + m) * B.rows + n] = acc;
        else
            put64(o, axes_offset(o.nr, o.rd, o.rs, (unsigned)m) + axes_offset(o.nc, o.cd, o.cs, (unsigned)n), acc);
    }
}
}  // namespace

double* small64(Ctx& c, const Operand64& A, const Operand64& B, const Out64& out, int& S) {
    const long long mt = (A.rows + ST - 1) / ST, nt = (B.rows + ST - 1) / ST;
    if (mt > 65535 || nt > 0x7fffffffLL || A.K >= (1LL << 30)) throw Error(-1, "small64: too many rows");
    const Small64Plan plan = plan_small64(mt * nt, A.K, sm_count());
    S = plan.S;
    double* T = out.p && S == 1 ? nullptr : c.arena.dalloc((size_t)S * A.rows * B.rows);
    k_small64<<<dim3((unsigned)nt, (unsigned)mt, (unsigned)S), ST * ST, 0, c.stream>>>(A, B, plan.terms, T, out);
    ++c.kernels;
    ADC_CUDA(cudaGetLastError());
    return T;
}

}  // namespace adc
