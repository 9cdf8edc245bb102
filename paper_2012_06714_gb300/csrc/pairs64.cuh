// FP64 ladder over pair-adapted integrals (pairs64.cu).
#pragma once
#include "common.cuh"

namespace adc {

// The pair-adapted integrals of ladder_tc.cuh to FP64 accuracy, as the digit planes of gemm64.
struct Pairs64 {
    int v = 0;
    long long P = 0, Pk = 0;
    Reclaimable store;  // digits of both halves
};

size_t pairs64_bytes(int nvir);
// forms them from B^Q_vv [naux][v][v]; false, holding nothing, if the device has no room
bool pairs64_prepare(Pairs64& L, Ctx& c, const double* Bvv, int naux, int nvir);
// out[n] += sum_Q B^Q X[n] B^Q for nmat matrices (store.mem[0] must be held)
void pairs64_apply(Pairs64& L, Ctx& c, const double* X, long long nmat, double* out);

}  // namespace adc
