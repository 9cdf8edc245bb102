// FP64-accurate contractions on the BF16 tensor cores of sm_103a (gemm64.cu).
#pragma once
#include <cuda_bf16.h>

#include "common.cuh"

namespace adc {

// A GEMM operand in its tensor's own storage: element (row, k) of the [rows][K] matrix lies at
// p[off_row(row) + off_k(k)], the offsets running over the row axes and the summed axes (row-major,
// `*_s` the strides of the tensor).
struct Operand64 {
    const void* p = nullptr;
    bool f32 = false;
    int nr = 0, nk = 0;
    long long rd[kMaxDim], rs[kMaxDim];  // row axes: extents, strides
    long long kd[kMaxDim], ks[kMaxDim];  // summed axes
    long long rows = 1, K = 1;
    void row_axis(long long d, long long s) { rd[nr] = d, rs[nr] = s, ++nr, rows *= d; }
    void k_axis(long long d, long long s) { kd[nk] = d, ks[nk] = s, ++nk, K *= d; }
};

// Whether gemm64 takes an M x N x K contraction rather than an FP64 kernel (sizes it is faster for).
bool gemm64_fits(long long M, long long N, long long K);

// C[M][N] = sum_k A[m][k] B[n][k] to FP64 accuracy.  With out: out[m][n] = alpha C + beta out, in one
// launch, when no K slices are needed (returns NULL).  Otherwise returns S results [S][M][N] in
// c.arena whose FP64 sum is C (without alpha and beta).  A bounded device wait that gives up raises
// c.d_err.
double* gemm64(Ctx& c, const Operand64& A, const Operand64& B, double alpha, double beta, double* out, int& S);

// A matrix already in digits: planes (one per digit, `plane` elements apart) of [rows][Kp] (Kp a
// multiple of 8, zeros beyond K) and the rows' exponents.
struct Digits64 {
    __nv_bfloat16* d = nullptr;
    int* ex = nullptr;
    long long rows = 0, Kp = 0, plane = 0;
};
size_t digits64_bytes(long long rows, long long K);  // of all planes
// one or two operands (of one Kp) into the caller's planes
void digitise64(Ctx& c, const Operand64* x, Digits64* out, int n);
// gemm64 of such matrices, never in place
double* gemm64_digits(Ctx& c, const Digits64& A, const Digits64& B, int& S);

}  // namespace adc
