// FP64 wavelength segments of Omega = u C on the log-log interpolant (Eq. interpolation), in fixed point where
// that is cheaper: shared by the exact build and the thermal-discrete rates.
#pragma once
#include "common.cuh"
#include "fix60.cuh"
#include "internal.h"

namespace heat {

// FP64 build: a segment's pieces, shared by every kernel of the exact path.  With Omega = u C, slope q - p - 1
// and Z = q dln, the segment's integral is v dln E1(Z) and up to the fraction tau of it v t E1(Z tau); E1 in 60-bit
// fixed point where |Z| < 1 (fix60.cuh; about 150 cycles of the integer pipes instead of 8 to 12 FP64
// multiply-adds of 64 cycles), else the library's expm1.
__device__ __forceinline__ double e1_of(double Z) {
    const int cls = e1_class(Z);
    return cls ? from_q60(e1_q60(cls, to_q60(Z))) : e1d(Z);
}
// Phi (Psi) after a segment: + v dln E1(Z)
__device__ __forceinline__ double add_segment(double sum, double v, double q, double dl) {
    return v > 0.0 ? fma(v * dl, e1_of(q * dl), sum) : sum;
}
struct SegF64 {
    double a, q1, aq;  // C_n u_n lambda_n^2 / h, slope + 2; a / q1 where the library's expm1 serves
    int64_t Z;         // q1 dln in Q60
    int cls;
    __device__ __forceinline__ SegF64(const GrainDev& gd, int g, int n, double ua, double su) {
        a = ua * gd.ca64[(size_t)g * gd.N + n];
        q1 = su + gd.sC[(size_t)g * gd.N + n] + 2.0;
        const double z = q1 * gd.dln[n];
        cls = e1_class(z);
        Z = cls ? to_q60(z) : 0;
        aq = cls ? 0.0 : a / q1;
    }
    // B at offset t (fraction tau) of the segment
    __device__ __forceinline__ double element(double Phi, double t, int64_t tau) const {
        if (cls) return fma(a * t, from_q60(e1_q60(cls, mul_q60(Z, tau))), Phi);
        return fma(aq, expm1(q1 * t), Phi);
    }
};
// The intra-bin term of a bin whose soft photons begin at offset t (fraction tau) of segment n, with Psi the
// integral of Omega beyond the segment: c (int from t to the segment's end + Psi) / (E_{j+1} - E_j).  The part of
// the segment is the difference of two fixed-point values, to 2^-53 of the whole segment's.
__device__ __forceinline__ double soft_term(const GrainDev& gd, int g, int n, double ua, double su, double t,
                                            int64_t tau, double Psi, double invdE) {
    const double b = ua * gd.ce64[(size_t)g * gd.N + n], q0 = su + gd.sC[(size_t)g * gd.N + n] + 1.0;
    const double dl = gd.dln[n], z = q0 * dl;
    double part = 0.0;
    if (b > 0.0) {
        const int cls = e1_class(z);
        if (cls) {
            const int64_t Z = to_q60(z);
            const int64_t d = e1_q60(cls, Z) - mul_q60(tau, e1_q60(cls, mul_q60(Z, tau)));
            part = d > 0 ? (b * dl) * from_q60(d) : 0.0;
        } else {
            const double L = dl - t;
            part = b * exp(q0 * t) * L * e1d(q0 * L);
        }
    }
    return __dmul_rn(__dmul_rn(kC, __dadd_rn(part, Psi)), invdE);
}
__device__ __forceinline__ double soft_end(double Psi, double invdE) { return __dmul_rn(__dmul_rn(kC, Psi), invdE); }

}  // namespace heat
