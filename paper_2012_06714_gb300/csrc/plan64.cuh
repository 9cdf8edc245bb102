// Launch plans of the FP64 contractions (gemm64.cu): host arithmetic only.
#pragma once

#include <algorithm>

namespace adc {

constexpr int GM = 128;   // tile rows
constexpr int GK = 32;    // K block: 64-byte rows, 64-byte swizzle
constexpr int EPOCH = 4;  // K blocks between drains (128 terms)

// A slice's sums are exact in 64 bits for up to 2^23 terms: the leading part of a result counts units of 2^88 in
// products of integers below 2^63, that is up to 2^38 for each term, and stays below 2^62.
constexpr int kExactBlocks = (1 << 23) / GK;

struct Gemm64Plan {
    int BNT, S, kb;  // tile width, K slices, K blocks per slice
};

// Tile width and K slices: least time over the chip.  A K block of a tile takes 18 BNT tensor cycles
// twice (36 digit pairs), reading A from shared memory bounds it below about BNT = 16; a drain (every
// EPOCH blocks) about 40 BNT cycles, which the MMAs wait for; the last one and the store about 60 BNT.
inline Gemm64Plan plan64(long long M, long long N, long long Kp, int sms) {
    const int num_k = (int)((Kp + GK - 1) / GK);
    if (num_k < 1) return Gemm64Plan{64, 1, EPOCH};
    const long long least = (num_k + kExactBlocks - 1) / kExactBlocks;
    Gemm64Plan p{64, (int)least, std::min(num_k, kExactBlocks)};
    double best = 1e300;
    for (int b : {64, 48, 32, 16}) {
        const long long tiles = std::max(1LL, ((M + GM - 1) / GM) * ((N + b - 1) / b));
        for (long long s = least; s <= std::max(1LL, std::min<long long>(160, 2 * sms / tiles)) || s <= least + 31; ++s) {
            const long long kb = ((num_k + s - 1) / s + EPOCH - 1) / EPOCH * EPOCH;
            if (kb > kExactBlocks || (s > 1 && (num_k + kb - 1) / kb != s)) continue;
            const double rounds = (double)((tiles * s + sms - 1) / sms);
            const double blocks = (double)std::min<long long>(kb, num_k);
            const double cyc = rounds * (2000.0 + blocks * 2.0 * std::max(18.0 * b, 320.0) + (blocks / EPOCH) * 40.0 * b + 60.0 * b) +
                               (s - 1) * (double)M * N * 16.0 / 2500.0 + (s > 1 ? 4000.0 : 0.0);
            if (cyc < best * 0.999) best = cyc, p = Gemm64Plan{b, (int)s, (int)kb};
        }
    }
    p.S = (num_k + p.kb - 1) / p.kb;
    return p;
}

// K slices of the kernel for the smallest contractions, and terms per slice: slices while the blocks leave SMs
// idle, of at least 64 terms (a sum of slices is another launch).
struct Small64Plan {
    int S;
    long long terms;
};
inline Small64Plan plan_small64(long long tiles, long long K, int sms) {
    Small64Plan p{1, std::max(1LL, K)};
    if (K >= 256 && tiles > 0 && tiles < 2 * sms) {
        p.S = (int)std::max<long long>(1, std::min<long long>({K / 64, 4LL * sms / tiles, 256}));
        p.terms = (K + p.S - 1) / p.S;
        p.S = (int)((K + p.terms - 1) / p.terms);
    }
    return p;
}

}  // namespace adc
