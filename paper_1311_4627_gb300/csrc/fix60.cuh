// E1(z) = (e^z - 1)/z in 60-bit fixed point (Q60: the value times 2^60) on the integer pipes, for the exact
// build.  In FP64 the Taylor series takes 8 to 12 multiply-adds of 64 cycles each; here the leading terms are
// 64-bit steps of three 32 x 32 multiply-adds, and the trailing ones, which the powers of z scale down,
// 32-bit steps.  Truncation and rounding are below 2^-53 of E1 on each range (2^-55.1 over 4000 arguments of each).
// Compiles for the host too (tests/test_fixed_point.py).
#pragma once
#include "isum.cuh"

namespace heat {

constexpr int64_t kQ60 = 1LL << 60;

// z (|z| <= 1) in Q60, truncated towards zero
HEAT_HD int64_t to_q60(double z) {
    const uint64_t b = bits64(z);
    const int e = (int)(b >> 52) & 0x7ff;
    const uint64_t m = ((b & 0xfffffffffffffull) | (e ? 0x10000000000000ull : 0ull)) << 8;  // 2^60 at exponent 1023
    const int64_t v = (int64_t)shr64(m, 1023 - e);
    return (int64_t)b < 0 ? -v : v;
}
// v > 0 in Q60 as the nearest double
HEAT_HD double from_q60(int64_t v) {
    const int lz = clz64((uint64_t)v);
    const uint64_t m = (uint64_t)v << lz, r = m + 0x400u;
    const int e = 1023 + 3 - lz + (r < m ? 1 : 0);
    return from_bits64(((uint64_t)e << 52) | ((r >> 11) & 0xfffffffffffffull));
}
// the Q60 product of two Q60 numbers below 2 in magnitude (to two units)
HEAT_HD int64_t mul_q60(int64_t a, int64_t b) {
    const int32_t ah = (int32_t)(a >> 30), al = (int32_t)(a & 0x3fffffff);
    const int32_t bh = (int32_t)(b >> 30), bl = (int32_t)(b & 0x3fffffff);
    return (int64_t)ah * bh + (((int64_t)ah * bl + (int64_t)al * bh) >> 30);
}

HEAT_HD constexpr double inv_factorial(int n) {
    double f = 1.0;
    for (int i = 2; i <= n; ++i) f /= i;
    return f;
}
// 2^60 / (k + 1)!, to the nearest integer
HEAT_HD constexpr int64_t e1_coef(int k) {
    int64_t f = 1;
    for (int i = 2; i <= k + 1; ++i) f *= i;
    return (kQ60 + f / 2) / f;
}
// sum_{k <= D} z^k / (k+1)!: terms above W in 32 bits, scaled by 2^S
template <int D, int W, int S>
HEAT_HD int64_t e1_series_q60(int64_t z) {
    const int32_t zh = (int32_t)(z >> 30), zl = (int32_t)(z & 0x3fffffff);
    int32_t q = (int32_t)(e1_coef(D) >> (30 - S));
#pragma unroll
    for (int k = D - 1; k > W; --k) q = (int32_t)(e1_coef(k) >> (30 - S)) + (int32_t)(((int64_t)q * zh) >> 30);
    int64_t p = e1_coef(W) + (((int64_t)q * zh) >> S);
#pragma unroll
    for (int k = W - 1; k >= 0; --k) {
        const int32_t ph = (int32_t)(p >> 30), pl = (int32_t)(p & 0x3fffffff);
        p = e1_coef(k) + (int64_t)ph * zh + (((int64_t)ph * zl + (int64_t)pl * zh) >> 30);
    }
    return p;
}
// The range that serves every |z| <= |Z|: 3: 1/16, 2: 1/4, 1: below 1, 0: none (the library's expm1).
HEAT_HD int e1_class(double Z) {
    const int e = (int)(bits64(Z) >> 52) & 0x7ff;  // |Z| < 2^(e - 1022)
    return e < 1019 ? 3 : e < 1021 ? 2 : e < 1023 ? 1 : 0;
}
HEAT_HD int64_t e1_q60(int cls, int64_t z) {
    return cls == 3 ? e1_series_q60<8, 4, 9>(z) : cls == 2 ? e1_series_q60<12, 6, 15>(z) : e1_series_q60<18, 10, 28>(z);
}

}  // namespace heat
