// FP64 contractions of sm_103a: exact digit products on the BF16 tensor cores, and a kernel of FP64
// arithmetic for the smallest ones (gemm64.cu).
#pragma once
#include <cuda_bf16.h>

#include "common.cuh"

namespace adc {

// A GEMM operand in its tensor's own storage: element (row, k) of the [rows][K] matrix lies at
// p[off_row(row) + off_k(k)], the offsets running over the row axes and the summed axes (row-major,
// `*s` the strides of the tensor).
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

// An operand in digits: planes (one per digit, `plane` elements apart) of [rows][Kp] (Kp a multiple of
// 8, zeros beyond K) and the rows' exponents.
struct Digits64 {
    __nv_bfloat16* d = nullptr;
    int* ex = nullptr;
    long long rows = 0, Kp = 0, plane = 0;
};
size_t digits64_bytes(long long rows, long long K);  // planes and exponents, in one buffer
Digits64 digits64_in(void* buffer, long long rows, long long K);
void digitise64(Ctx& c, const Operand64* x, Digits64* out, int n);  // one or two operands (of one Kp)

// Where a result goes: out[off_row(m) + off_col(n)] = alpha C + beta out (axes as in Operand64, the
// rows those of A, the columns those of B).
struct Out64 {
    double* p = nullptr;
    double alpha = 1.0, beta = 0.0;
    int nr = 0, nc = 0;
    long long rd[kMaxDim], rs[kMaxDim], cd[kMaxDim], cs[kMaxDim];
    void row_axis(long long d, long long s) { rd[nr] = d, rs[nr] = s, ++nr; }
    void col_axis(long long d, long long s) { cd[nc] = d, cs[nc] = s, ++nc; }
};

// C[M][N] = sum_k A[m][k] B[n][k] in FP64.  Written to `out` in the same launch when no K slices are
// needed (returns NULL); otherwise, or with out.p NULL, returns S results [S][M][N] in c.arena whose
// sum is C.  gemm64 works on the tensor cores and takes operands in digits (da, db: else made here);
// a bounded device wait that gives up raises c.d_err.  small64 works in FP64 arithmetic.
bool gemm64_fits(long long M, long long N, long long K);  // sizes it is the faster one for
double* gemm64(Ctx& c, const Operand64& A, const Digits64* da, const Operand64& B, const Digits64* db, const Out64& out,
               int& S);
double* small64(Ctx& c, const Operand64& A, const Operand64& B, const Out64& out, int& S);

}  // namespace adc
