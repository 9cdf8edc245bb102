// The ladder sum_cd (ac|bd) X_n[c,d] to FP64 accuracy: the contraction over symmetric and
// antisymmetric pairs of ladder_tc.cu with the integrals, the vectors and the products of gemm64.
//
// nmat v^4 flops on the tensor cores instead of 4 naux v^3 nmat on the FP64 units through two DGEMMs
// per auxiliary function (which stay for the sizes whose integrals do not fit: 32 P^2 bytes, P = v (v +
// 1) / 2, i.e. 0.7 GB at v = 97, 8.5 GB at 180).  Bound by reading the integrals' digits (16 bytes each)
// for few matrices, by the tensor cores beyond about 40.
// Measured, FP64 sigma of 4 vectors at 12/97/381: 142 -> 0.73 ms (the ladder 129 -> 0.25 ms, both halves'
// 361 MB of digits at 3.5 TB/s), its error against 64 bits 9.2e-16 -> 1.7e-16; four roots at 8/45/187:
// 165 -> 7.6 ms.
#include "pairs64.cuh"

#include <algorithm>

#include "gemm64.cuh"
#include "pairs.cuh"

namespace adc {
namespace {

struct PutDoubles {
    double* o;  // [2][rows][P]
    long long rows, P, row0;
    __device__ void operator()(int half, long long row, long long p, double x) const { o[(half * rows + row) * P + p] = x; }
    __device__ void pad(long long, int) const {}
};

Operand64 rows_of(const double* p, long long rows, long long K) {
    Operand64 o;
    o.p = p;
    o.row_axis(rows, K);
    o.k_axis(K, 1);
    return o;
}

// digits of one half of L, rows [row0, row0 + rows)
Digits64 half_of(const Pairs64& L, int half, long long row0, long long rows) {
    Digits64 d = digits64_in((char*)L.store.mem[0] + half * digits64_bytes(L.P, L.P), L.P, L.P);
    d.rows = rows;
    d.d += row0 * L.Pk;
    d.ex += row0;
    return d;
}

}  // namespace

size_t pairs64_bytes(int v) {
    const long long P = (long long)v * (v + 1) / 2;
    return 2 * digits64_bytes(P, P);
}

bool pairs64_prepare(Pairs64& L, Ctx& c, const double* Bvv, int naux, int nvir) {
    const long long v = nvir, Q = naux, P = v * (v + 1) / 2;
    if (P >= (1LL << 30) || v * v >= (1LL << 30)) return false;
    void* base = nullptr;
    if (dev_malloc_raw(&base, pairs64_bytes(nvir), c.stream) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    L.v = nvir;
    L.P = P;
    L.Pk = (P + 7) / 8 * 8;
    ReclaimPin pin(L.store, c.stream);  // its own allocations may not take them away again
    L.store.hold(base, nullptr, pin);
    // rows (a, c) of a block of a's against the columns (b, d), b <= the block's last a: at most 1 GB,
    // packed into the pairs' rows a (a + 1) / 2 + b and cut into digits
    for (long long a0 = 0; a0 < v;) {
        long long na = 1;
        while (a0 + na < v && (na + 1) * v * (a0 + na + 1) * v * 8 <= (1LL << 30)) ++na;
        const long long nb = a0 + na, r0 = a0 * (a0 + 1) / 2, rows = nb * (nb + 1) / 2 - r0;
        Arena::Mark mk = c.arena.mark();
        Operand64 A, B;
        A.p = Bvv + a0 * v;
        A.row_axis(na, v);
        A.row_axis(v, 1);
        A.k_axis(Q, v * v);
        B.p = Bvv;
        B.row_axis(nb, v);
        B.row_axis(v, 1);
        B.k_axis(Q, v * v);
        double* G = c.arena.dalloc((size_t)(na * v * nb * v));
        int S = 1;
        Out64 go;
        go.p = G;
        go.row_axis(na * v, nb * v);
        go.col_axis(nb * v, 1);
        const double* T = gemm64(c, A, nullptr, B, nullptr, go, S);
        if (T) {
            Shape sh{1, {na * v * nb * v}};
            const int id[1] = {0};
            permute_sum(c, T, S, sh, id, G, false, 1.0, 0.0);
        }
        double* VP = c.arena.dalloc((size_t)(2 * rows * P));
        const long long nt = (v + 31) / 32, tiles = na * nb * nt * (nt + 1) / 2;
        k_pair_pack<double, PutDoubles><<<(unsigned)std::min<long long>(tiles, 152LL * 16), dim3(32, 8), 0, c.stream>>>(
            G, (int)v, na * nb, 0, nb * v, 1, (int)a0, (int)nb, PutDoubles{VP, rows, P, r0});
        ++c.kernels;
        ADC_CUDA(cudaGetLastError());
        const Operand64 x[2] = {rows_of(VP, rows, P), rows_of(VP + rows * P, rows, P)};
        Digits64 d[2] = {half_of(L, 0, r0, rows), half_of(L, 1, r0, rows)};
        digitise64(c, x, d, 2);
        c.arena.release(mk);
        a0 += na;
    }
    return true;
}

void pairs64_apply(Pairs64& L, Ctx& c, const double* X, long long nmat, double* out) {
    const long long v = L.v, P = L.P;
    // groups of matrices whose pairs, digits and results (16, 32 and about 32 P bytes each) stay within 4 GiB
    const long long mg = std::max<long long>(1, std::min<long long>(nmat, (4LL << 30) / (80 * P)));
    ReclaimPin pin(L.store, c.stream);
    for (long long m0 = 0; m0 < nmat; m0 += mg) {
        const long long nm = std::min(mg, nmat - m0);
        Arena::Mark mk = c.arena.mark();
        double* XP = c.arena.dalloc((size_t)(2 * nm * P));
        const long long nt = (v + 31) / 32, tiles = nm * nt * (nt + 1) / 2;
        k_pair_pack<double, PutDoubles><<<(unsigned)std::min<long long>(tiles, 152LL * 16), dim3(32, 8), 0, c.stream>>>(
            X + m0 * v * v, (int)v, nm, v * v, v, 0, 0, 1, PutDoubles{XP, nm, P, 0});
        ++c.kernels;
        ADC_CUDA(cudaGetLastError());
        const Operand64 x[2] = {rows_of(XP, nm, P), rows_of(XP + nm * P, nm, P)};
        Digits64 d[2];
        for (int h = 0; h < 2; ++h) d[h] = digits64_in(c.arena.alloc(digits64_bytes(nm, P)), nm, P);
        digitise64(c, x, d, 2);
        int S = 1;
        const Operand64 none{};
        const Digits64 V0 = half_of(L, 0, 0, P), V1 = half_of(L, 1, 0, P);
        const double* T0 = gemm64(c, none, &V0, none, &d[0], Out64(), S);
        const double* T1 = gemm64(c, none, &V1, none, &d[1], Out64(), S);
        const long long ut = (v + 15) / 16, blocks = ut * (ut + 1) / 2 * ((nm + 7) / 8);
        k_pair_unfold<double><<<(unsigned)std::min<long long>(blocks, 152LL * 32), 256, 0, c.stream>>>(
            T0, T1, S, P, (int)nm, (int)v, out + m0 * v * v);
        ++c.kernels;
        ADC_CUDA(cudaGetLastError());
        c.arena.release(mk);
    }
}

}  // namespace adc
