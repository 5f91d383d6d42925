// Sums of products of non-negative numbers in 64-bit fixed point, on the integer pipes.
//
// A GB300 sub-partition's FP64 unit takes 64 cycles per warp-wide multiply-add; its integer pipes take
// 2.3 cycles per 32-bit operation and 4.8 per 32 x 32 + 64-bit multiply-add (measured).  A product of two
// mantissas, aligned to the largest term of the sum and added in 64 bits, is about 25 cycles of them.
// Every term is non-negative, so nothing cancels: a term is kept to 2^-61 of the largest one (dropped bits
// only below that), against FP64's rounding to 2^-53 of the running sum at every addition.  Exponents are
// plain integers: nothing overflows or underflows between the operands and the rounded result.
//
// Compiles for the host too (tests/test_fixed_point.py checks the arithmetic there).
#pragma once
#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>

namespace heat {

#define HEAT_HD __host__ __device__ __forceinline__

// a >> d, 0 for d > 63 (d >= 0)
HEAT_HD uint64_t shr64(uint64_t a, int d) {
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(d));
    return r;
#else
    return d > 63 ? 0 : a >> d;
#endif
}
HEAT_HD int clz64(uint64_t a) {  // a != 0
#ifdef __CUDA_ARCH__
    return __clzll((long long)a);
#else
    return __builtin_clzll(a);
#endif
}
constexpr uint64_t kMag64 = 0x7fffffffffffffffull;  // all but the sign (a -0 counts as 0)
HEAT_HD uint64_t bits64(double x) {
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t b;
    std::memcpy(&b, &x, 8);
    return b;
#endif
}
HEAT_HD double from_bits64(uint64_t b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double x;
    std::memcpy(&x, &b, 8);
    return x;
#endif
}
// A double x >= 0 as mantissa (h, l) with the leading bit at bit 63 and biased exponent e; 0 has mantissa 0 and an
// exponent below every other, so that it raises no sum's exponent.  x = (h:l) 2^(e - 1086).
constexpr int kZeroExp = 4096;
struct Mant {
    uint32_t h, l;
    int e;
};
HEAT_HD Mant mant(double x) {
    const uint64_t b = bits64(x) & kMag64;
    const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
    Mant r;
    r.e = (int)(hi >> 20);
    r.h = (hi << 11) | (lo >> 21) | 0x80000000u;
    r.l = lo << 11;
    if (r.e == 0) {  // zero, or subnormal: normalised
        const int lz = b ? clz64(b) : 0;
        const uint64_t m = b << lz;
        r.h = (uint32_t)(m >> 32);
        r.l = (uint32_t)m;
        r.e = b ? 12 - lz : -kZeroExp;
    }
    return r;
}
// a b as a 64-bit product p and exponent ep: value p 2^(ep - kProdExp); the low parts' product is below 2^-64 of the
// whole and left out
constexpr int kProdExp = 2108;
HEAT_HD void mul(const Mant& a, const Mant& b, uint64_t& p, int& ep) {
    p = (uint64_t)a.h * b.h + (((uint64_t)a.h * b.l) >> 32) + (((uint64_t)a.l * b.h) >> 32);
    ep = a.e + b.e;
}

// The sum: value a 2^(E + 3 - kProdExp).  Terms enter shifted to the exponent E (the largest so far) with three
// bits of headroom.
struct ISum {
    uint64_t a = 0;
    int E = -100000;
    HEAT_HD void raise(int En) {  // En >= E
        a = shr64(a, En - E);
        E = En;
    }
    HEAT_HD void settle() {  // after at most four terms: below 2^62 again
        if ((int64_t)a < 0) {
            a >>= 2;
            E += 2;
        }
    }
    // rounded to the nearest double (infinity beyond the range)
    HEAT_HD double value() const {
        if (a == 0) return 0.0;
        const int lz = clz64(a);
        uint64_t m = a << lz;
        int e = E - lz + 1089 - kProdExp;
        if (e <= 0) return from_bits64((shr64(m, 11 - e) + 1) >> 1);  // below the normal range: to a multiple of 2^-1074
        m += 0x400u;  // half of a unit in the 53rd place (ties away from zero)
        const uint64_t carry = m < 0x400u ? 1u : 0u;  // all ones: the next power of two
        e += (int)carry;
        // the leading bit adds 1 to the exponent field
        const uint64_t r = carry ? 0 : (m >> 11) & 0x000fffffffffffffull;
        return from_bits64(e < 2047 ? ((uint64_t)e << 52) | r : 0x7ff0000000000000ull);
    }
};

// Four consecutive values >= 0 aligned to the largest of them: x[u] = (h[u] 2^27 + l[u]) 2^(E - 1079), 30 and
// 27 bits; what is dropped is below 2^-57 of the largest.
struct Align4 {
    uint32_t h[4], l[4];
    int E;
};
HEAT_HD Align4 align4(const double (&x)[4]) {
    Align4 r;
    int e[4];
    for (int u = 0; u < 4; ++u) {
        e[u] = (int)((bits64(x[u]) & kMag64) >> 52);
        e[u] += e[u] == 0;  // zeros and subnormals: the exponent of the smallest normal, no leading bit
    }
    const int a = e[0] > e[1] ? e[0] : e[1], b = e[2] > e[3] ? e[2] : e[3];
    r.E = a > b ? a : b;
    for (int u = 0; u < 4; ++u) {
        const uint64_t lead = (bits64(x[u]) & 0x7ff0000000000000ull) ? 0x10000000000000ull : 0ull;
        const uint64_t v = (bits64(x[u]) & 0xfffffffffffffull) | lead;
        const uint64_t y = shr64(v << 4, r.E - e[u]);
        r.h[u] = (uint32_t)(y >> 27);
        r.l[u] = (uint32_t)y & 0x7ffffffu;
    }
    return r;
}
// s += sum_u a[u] b[u] of aligned fours (FP64 sums' scale): the products are added by the multiply-adds
// themselves and brought to the sum's exponent once.
HEAT_HD void add_aligned4(ISum& s, const uint32_t (&ah)[4], const uint32_t (&al)[4], int aE, const uint32_t (&bh)[4],
                          const uint32_t (&bl)[4], int bE) {
    uint64_t H = 0, C = 0;
    for (int u = 0; u < 4; ++u) {
        H += (uint64_t)ah[u] * bh[u];
        C += (uint64_t)ah[u] * bl[u];
        C += (uint64_t)al[u] * bh[u];
    }
    const uint64_t t = H + (C >> 27);  // below 2^62 + 2^34; value t 2^(aE + bE - 2104)
    const int ep = t ? aE + bE + 1 : -100000;
    const int En = s.E > ep ? s.E : ep;
    s.raise(En);
    s.a += shr64(t, En - ep);
    s.settle();
}
// the same one by one (operands of very different size among the four)
HEAT_HD void add_each4(ISum& s, const Mant (&a)[4], const Mant (&b)[4]) {
    uint64_t p[4];
    int ep[4], En = s.E;
    for (int u = 0; u < 4; ++u) {
        mul(a[u], b[u], p[u], ep[u]);
        En = En > ep[u] ? En : ep[u];
    }
    s.raise(En);
    for (int u = 0; u < 4; ++u) s.a += shr64(p[u], En - ep[u] + 3);
    s.settle();
}

}  // namespace heat
