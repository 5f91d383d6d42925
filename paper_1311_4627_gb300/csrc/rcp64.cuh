// FP64 reciprocal with three FP64 operations, for the state reduction's serial chain (k_discrete.cu).
#pragma once
#include <cuda_runtime.h>

namespace heat {

// Reciprocal of x >= 0 (0 for 0): for a mantissa m in [1, 2) the hardware's FP32 reciprocal y of its leading
// bits (relative error e = 1 - m y < 2^-21), then y + y (e + e^2), whose error e^3 is below 2^-63, so that the result
// is off by half an ulp and 2^-10 of one.  Three dependent FP64 operations of 64 cycles where a division has eight.
__device__ __forceinline__ double rcp_or_0(double x) {
    const int h = __double2hiint(x), l = __double2loint(x), ex = h >> 20;
    if ((unsigned)(ex - 64) > 1900u) return x > 0.0 ? 1.0 / x : 0.0;  // zero, subnormal, very large, infinite
    const double m = __hiloint2double((h & 0xfffff) | 0x3ff00000, l);
    float yf;
    asm("rcp.approx.ftz.f32 %0, %1;"
        : "=f"(yf)
        : "f"(__uint_as_float(0x3f800000u | ((unsigned)(h & 0xfffff) << 3) | ((unsigned)l >> 29))));
    const unsigned fb = __float_as_uint(yf);
    double y = __hiloint2double((int)((fb >> 3) + 0x38000000u), (int)(fb << 29));
    const double e = fma(-m, y, 1.0);
    y = fma(y, fma(e, e, e), y);
    return __hiloint2double(__double2hiint(y) + ((1023 - ex) << 20), __double2loint(y));
}

}  // namespace heat
