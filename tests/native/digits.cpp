// The host side of gemm64.cu's arithmetic (digits.cuh, plan64.cuh): digit products of rows over the whole range
// of doubles against long double sums, the 64-bit sums at the longest slice, and launch plans at their ends.
#include <cfloat>
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "digits.cuh"
#include "plan64.cuh"

using namespace adc;

static int bad = 0;
#define CHECK(x, ...)                                                        \
    do {                                                                     \
        if (!(x) && bad++ < 20) std::printf("line %d: %s  ", __LINE__, #x), std::printf(__VA_ARGS__), std::printf("\n"); \
    } while (0)

static uint64_t bits_of(double x) {
    uint64_t b;
    std::memcpy(&b, &x, sizeof b);
    return b;
}

// sum_k a_k b_k the way the kernels form it
static double product(const std::vector<double>& a, const std::vector<double>& b) {
    int ea = 0, eb = 0;
    for (double x : a) ea = std::max(ea, exponent_of(bits_of(x)));
    for (double x : b) eb = std::max(eb, exponent_of(bits_of(x)));
    long long hi = 0, lo = 0;
    for (size_t k = 0; k < a.size(); ++k) {
        const long long va = scaled_integer(bits_of(a[k]), ea), vb = scaled_integer(bits_of(b[k]), eb);
        const uint64_t wa = with_carries(va), wb = with_carries(vb);
        long long s[NL] = {};
        for (int i = 0; i < ND; ++i)
            for (int j = 0; j < ND; ++j)
                if (i + j >= SMIN) s[i + j - SMIN] += (long long)digit(va, wa, i) * digit(vb, wb, j);
        hi += s[7] * (1 << 24) + s[6] * (1 << 16) + s[5] * (1 << 8) + s[4];
        lo += s[3] * (1 << 24) + s[2] * (1 << 16) + s[1] * (1 << 8) + s[0];
    }
    return to_double(hi, lo, 8 * SMIN + ea + eb - 2 * 1085);
}

int main() {
    std::mt19937_64 g(1);
    std::normal_distribution<double> n01;
    // digits add up to their integer
    for (int i = 0; i < 200000; ++i) {
        long long v = (long long)(g() >> (1 + g() % 62));
        if (i < 4) v = i < 2 ? 0x7ffffffffffffc00LL - i : (1LL << 55) - 128 + i;
        if (g() & 1) v = -v;
        const uint64_t w = with_carries(v);
        __int128 sum = 0;
        for (int p = ND - 1; p >= 0; --p) {
            const int d = digit(v, w, p);
            CHECK(d >= -128 && d <= 128, "%lld digit %d = %d", v, p, d);
            sum = sum * 256 + d;
        }
        CHECK(sum == v, "%lld", v);
    }
    // products of rows of any size: the stated bound, one rounding to FP64, one unit of the subnormal numbers
    for (int i = 0; i < 4000; ++i) {
        const int K = 1 + (int)(g() % 300);
        const int pa = i % 4 == 0 ? -1040 - (int)(g() % 34) : -500 + (int)(g() % 1000);  // subnormal rows too
        const int pb = i % 4 == 0 ? (int)(g() % 900) : i % 4 == 1 ? -1010 - pa + (int)(g() % 5) : -400 + (int)(g() % 800);
        std::vector<double> a(K), b(K);
        long double exact = 0, ma = DBL_MIN, mb = DBL_MIN;
        for (int k = 0; k < K; ++k) {
            a[k] = std::ldexp(n01(g), pa - (i % 3 ? 0 : (int)(g() % 60)));
            b[k] = std::ldexp(n01(g), pb);
            exact += (long double)a[k] * b[k];
            ma = std::fmax(ma, std::fabs((long double)a[k])), mb = std::fmax(mb, std::fabs((long double)b[k]));
        }
        const double r = product(a, b);
        // (2 ma and 2 mb: the rows' powers of two, at least that of the smallest normal numbers; long double
        // sums carry 2^-64 K of their own)
        const long double allowed = fabsl(exact) * 0x1p-53L + K * 4 * ma * mb * 0x1.1p-61L + 0x1p-1074L;
        CHECK(fabsl((long double)r - exact) <= allowed, "K %d, 2^%d 2^%d: %a, exact %La", K, pa, pb, r, exact);
    }
    // a slice of constant rows at their largest: the leading part within 62 bits, the sum exact
    {
        const long long terms = (long long)kExactBlocks * GK, v = 0x7ffffffffffffc00LL;
        const uint64_t w = with_carries(v);
        __int128 hi = 0, lo = 0;
        for (int i = 0; i < ND; ++i)
            for (int j = SMIN - i; j < ND; ++j) {
                const __int128 d = (__int128)digit(v, w, i) * digit(v, w, j) * terms;
                (i + j >= 11 ? hi : lo) += d << (8 * (i + j >= 11 ? i + j - 11 : i + j - SMIN));
            }
        const __int128 lim = (__int128)1 << 62;
        CHECK(hi < lim && hi > -lim && lo < lim && lo > -lim, "%d terms", (int)terms);
    }
    // the ends of the range of results
    CHECK(to_double((1LL << 53) - 1, 0, 971 - 32) == DBL_MAX, "%a", to_double((1LL << 53) - 1, 0, 971 - 32));
    CHECK(to_double(0, 3, 1022) == 0x1.8p+1023, "%a", to_double(0, 3, 1022));
    CHECK(std::isinf(to_double(1, 0, 1024 - 32)), " ");
    CHECK(to_double(0, -1, -1074) == -0x1p-1074, " ");
    CHECK(to_double(0, 5, -1073) == 0xap-1074, " ");
    CHECK(to_double(0, 1, -1076) == 0.0, " ");
    CHECK(to_double(0, 0, 0) == 0.0, " ");
    // plans: every K block in one slice, no empty slice, no slice beyond the exact sums
    for (int i = 0; i < 20000; ++i) {
        auto size = [&](int top) { return (long long)std::exp2(std::uniform_real_distribution<double>(0, top)(g)); };
        const long long M = i < 8 ? i % 2 : size(24), N = i < 8 ? i / 2 % 2 : size(24);
        const long long Kp = i < 8 ? i / 4 * 8 : (size(27) + 7) / 8 * 8 << (i % 5 == 0 ? 2 : 0);
        const Gemm64Plan p = plan64(M, N, Kp, 152);
        const long long num_k = (Kp + GK - 1) / GK;
        CHECK(p.S >= 1 && (long long)p.S * p.kb >= num_k && (p.S == 1 || (p.S - 1LL) * p.kb < num_k), "%lld %lld %lld", M, N, Kp);
        CHECK(p.kb <= kExactBlocks && (p.S == 1 || p.kb % EPOCH == 0), "%lld: %d slices of %d", Kp, p.S, p.kb);
        const long long tiles = i < 8 ? i % 2 : size(20), K = i < 8 ? i / 2 : size(22);
        const Small64Plan q = plan_small64(tiles, K, 152);
        CHECK(q.S >= 1 && q.S * q.terms >= K && (q.S == 1 || (q.S - 1) * q.terms < K), "%lld %lld", tiles, K);
    }
    if (bad) std::printf("%d wrong\n", bad);
    return bad ? 1 : 0;
}
