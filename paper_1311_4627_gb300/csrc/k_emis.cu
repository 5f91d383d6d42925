// Emissivity contraction (Eq. emission, Eq. emission-lambda) in FP64:
//   j[c][g][n] = sum_i P[c][off_g + i] K[off_g + i][n],   K = C_abs B_lambda(T_i) [E_i >= hc/lambda_n],
// and the size-integrated form over the concatenated bins with K scaled by w_g (Eq. convolution).
// Three forms: sums in 64-bit fixed point on the integer pipes (k_gemm_i64), a register-tiled SIMT
// GEMM on the FP64 FMA pipe for kernels that may be negative, and a thread per output for few rows.
#include "common.cuh"
#include "internal.h"
#include "isum.cuh"

namespace heat {

template <typename TC>
__global__ void __launch_bounds__(256, 2) k_gemm_f64(int M, int N, const int* __restrict__ koff,
                                                  const double* __restrict__ A, long long lda,
                                                  const double* __restrict__ B, long long ldb, TC* __restrict__ C,
                                                  long long ldc, long long zs) {
    __shared__ double As[16][65];
    __shared__ double Bs[16][64];
    const int z = blockIdx.z;
    const int k0 = koff[z], k1 = koff[z + 1];
    const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    double acc[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int s = 0; s < 4; ++s) acc[r][s] = 0.0;
    for (int kb = k0; kb < k1; kb += 16) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            int idx = tid + 256 * r;
            int mm = idx >> 4, kk = idx & 15;
            double v = 0.0;
            if (m0 + mm < M && kb + kk < k1) v = A[(size_t)(m0 + mm) * lda + kb + kk];
            As[kk][mm] = v;
            int kr = idx >> 6, nn = idx & 63;
            double w = 0.0;
            if (kb + kr < k1 && n0 + nn < N) w = B[(size_t)(kb + kr) * ldb + n0 + nn];
            Bs[kr][nn] = w;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            double a[4], b[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) a[r] = As[kk][ty + 16 * r];
#pragma unroll
            for (int s = 0; s < 4; ++s) b[s] = Bs[kk][tx + 16 * s];
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int s = 0; s < 4; ++s) acc[r][s] = fma(a[r], b[s], acc[r][s]);
        }
        __syncthreads();
    }
    TC* Cz = C + (size_t)z * zs;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        int m = m0 + ty + 16 * r;
        if (m >= M) continue;
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            int n = n0 + tx + 16 * s;
            if (n < N) Cz[(size_t)m * ldc + n] = (TC)acc[r][s];
        }
    }
}

// One output's FMA chain, for columns that fixed point cannot hold (an infinite K).
__device__ __noinline__ double chain_f64(int k0, int k1, const double* a, const double* b, long long ldb) {
    double acc = 0.0;
    for (int k = k0; k < k1; ++k) acc = fma(a[k], b[(size_t)k * ldb], acc);
    return acc;
}

// The contraction of non-negative operands without the FP64 unit, which takes 64 cycles per warp-wide
// multiply-add: the sums run in 64-bit fixed point on the integer pipes (isum.cuh), four bins at a time.
//   * Four bins whose K values lie within a factor of 2^4 in every column of the tile: both operands are
//     aligned to the largest of their four (at staging, once per 32 or 64 outputs), a product is three
//     multiply-adds, and one shift per four products brings them to the sum's exponent: about 18 cycles a
//     product.  What a four drops is below 17 x 2^-58 of its largest operands' product.
//   * Otherwise (the Wien side, where K climbs steeply) each product is aligned by itself: 36 cycles.
//   * Four bins without any emission in the tile's columns (K = 0: the bin's energy or temperature is too low)
//     are left out.
// Which form a column's bins take depends on K alone, so a cell's result does not depend on the others'.
// Errors are below the FMA chain's (each row is rounded to FP64 once).  Measured at 512 cells x 64 grains x
// 1024 wavelengths (36864 bins): 31.3 -> 10.7 ms; both operands are staged in the one form that their four takes (in both,
// 11.3 ms).
// Tile 64 rows x 32 columns per 256 threads, 4 x 2 outputs a thread, 16 bins staged at a time.
template <typename TC>
__global__ void __launch_bounds__(256, 2) k_gemm_i64(int M, int N, const int* __restrict__ koff,
                                                     const double* __restrict__ A, long long lda,
                                                     const double* __restrict__ B, long long ldb, TC* __restrict__ C,
                                                     long long ldc, long long zs) {
    constexpr int KB = 4;  // fours of bins per stage
    __shared__ uint4 Ah[KB][64], Al[KB][64], Bh[KB][32], Bl[KB][32];
    __shared__ int Ae[KB][64], Be[KB][32];
    __shared__ Mant Am[KB][4][64], Bm[KB][4][32];  // for the one-by-one form
    __shared__ int flag[KB];  // 0: no emission, 1: aligned, 3: one by one
    __shared__ int bad[64];   // rows with a NaN or an infinity
    __shared__ int badc[32];  // columns with an infinity (or a NaN)
    const int z = blockIdx.z;
    const int k0 = koff[z], k1 = koff[z + 1];
    const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 32;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    if (tid < 64) bad[tid] = 0;
    if (tid < 32) badc[tid] = 0;
    ISum S[4][2];
    for (int kb = k0; kb < k1; kb += 4 * KB) {
        if (tid < KB) flag[tid] = 0;
        __syncthreads();
        if (tid < 32 * KB) {
            const int c = tid & 31, q = tid >> 5, n = n0 + c;
            double x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = kb + 4 * q + u;
                x[u] = (k < k1 && n < N) ? B[(size_t)k * ldb + n] : 0.0;
            }
            // compared as integers: the values are not negative (the FP64 unit takes 64 cycles a comparison)
            const int kn = k1 - (kb + 4 * q);  // bins of this four
            long long lo = (long long)(bits64(x[0]) & kMag64), hi = lo;
#pragma unroll
            for (int u = 1; u < 4; ++u)
                if (u < kn) {
                    lo = min(lo, (long long)(bits64(x[u]) & kMag64));
                    hi = max(hi, (long long)(bits64(x[u]) & kMag64));
                }
            if (hi >= 0x7ff0000000000000ll) badc[c] = 1;
            const int f = hi > 0 ? (hi - lo > (3LL << 52) ? 3 : 1) : 0;  // (a difference of 3 exponents: 2^3 to 2^4)
            const int any = __reduce_or_sync(0xffffffffu, f);
            if (any == 1) {  // only the form that the four's columns take
                const Align4 a = align4(x);
                Bh[q][c] = make_uint4(a.h[0], a.h[1], a.h[2], a.h[3]);
                Bl[q][c] = make_uint4(a.l[0], a.l[1], a.l[2], a.l[3]);
                Be[q][c] = a.E;
            } else if (any) {
#pragma unroll
                for (int u = 0; u < 4; ++u) Bm[q][u][c] = mant(x[u]);
            }
            if (c == 0) flag[q] = any;
        }
        __syncthreads();
        // nothing to add (the last stage is kept: it carries a row's NaN into columns without emission)
        if ((flag[0] | flag[1] | flag[2] | flag[3]) == 0 && kb + 4 * KB < k1) continue;
        {
            const int r = tid >> 2, q = tid & 3, m = m0 + r;  // consecutive threads: consecutive fours of a row
            double x[4];
            bool nan = false;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = kb + 4 * q + u;
                x[u] = (m < M && k < k1) ? A[(size_t)m * lda + k] : 0.0;
                nan |= (__double2hiint(x[u]) & 0x7ff00000) == 0x7ff00000;
            }
            const int f = flag[q];
            if (f == 1) {
                const Align4 a = align4(x);
                Ah[q][r] = make_uint4(a.h[0], a.h[1], a.h[2], a.h[3]);
                Al[q][r] = make_uint4(a.l[0], a.l[1], a.l[2], a.l[3]);
                Ae[q][r] = a.E;
            } else if (f) {
#pragma unroll
                for (int u = 0; u < 4; ++u) Am[q][u][r] = mant(x[u]);
            }
            if (nan) bad[r] = 1;
        }
        __syncthreads();
#pragma unroll 1
        for (int q = 0; q < KB; ++q) {
            const int f = flag[q];
            if (f == 1) {
                uint32_t bh[2][4], bl[2][4];
                int be[2];
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    const uint4 h = Bh[q][tx + 16 * s], l = Bl[q][tx + 16 * s];
                    bh[s][0] = h.x, bh[s][1] = h.y, bh[s][2] = h.z, bh[s][3] = h.w;
                    bl[s][0] = l.x, bl[s][1] = l.y, bl[s][2] = l.z, bl[s][3] = l.w;
                    be[s] = Be[q][tx + 16 * s];
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const uint4 h = Ah[q][ty + 16 * r], l = Al[q][ty + 16 * r];
                    const uint32_t ah[4] = {h.x, h.y, h.z, h.w}, al[4] = {l.x, l.y, l.z, l.w};
                    const int ae = Ae[q][ty + 16 * r];
#pragma unroll
                    for (int s = 0; s < 2; ++s) add_aligned4(S[r][s], ah, al, ae, bh[s], bl[s], be[s]);
                }
            } else if (f) {
                Mant b[2][4];
#pragma unroll
                for (int s = 0; s < 2; ++s)
#pragma unroll
                    for (int u = 0; u < 4; ++u) b[s][u] = Bm[q][u][tx + 16 * s];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    Mant a[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) a[u] = Am[q][u][ty + 16 * r];
#pragma unroll
                    for (int s = 0; s < 2; ++s) add_each4(S[r][s], a, b[s]);
                }
            }
        }
        __syncthreads();
    }
    TC* Cz = C + (size_t)z * zs;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int m = m0 + ty + 16 * r;
        if (m >= M) continue;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int n = n0 + tx + 16 * s;
            if (n >= N) continue;
            double v = S[r][s].value();
            if (bad[ty + 16 * r]) v = NAN;
            if (badc[tx + 16 * s]) v = chain_f64(k0, k1, A + (size_t)m * lda, B + n, ldb);
            Cz[(size_t)m * ldc + n] = (TC)v;
        }
    }
}

// Solves of few cells: a thread per output, threads along n (coalesced rows of K), one accumulator in
// ascending k (k_gemm_f64's bits; k_gemm_i64's sums are rounded once and differ in the last bits); the
// 64-row tiles above would spend 64 products per useful one on a single cell.
template <typename TC>
__global__ void __launch_bounds__(128) k_gemv_f64(int N, const int* __restrict__ koff, const double* __restrict__ A,
                                                  long long lda, const double* __restrict__ B, long long ldb,
                                                  TC* __restrict__ C, long long ldc, long long zs) {
    const int z = blockIdx.z, m = blockIdx.y, n = blockIdx.x * 128 + threadIdx.x;
    if (n >= N) return;
    const int k0 = koff[z], k1 = koff[z + 1];
    const double* a = A + (size_t)m * lda;
    double acc = 0.0;
    for (int k = k0; k < k1; ++k) acc = fma(a[k], B[(size_t)k * ldb + n], acc);
    C[(size_t)z * zs + (size_t)m * ldc + n] = (TC)acc;
}

cudaError_t launch_gemm_f64(int M, int N, int nz, const int* koff, const double* A, long long lda, const double* B,
                            long long ldb, void* C, long long ldc, long long zstride_c, int c_is_f32, int b_nonneg,
                            int few, cudaStream_t st) {
    if (M <= 0 || N <= 0 || nz <= 0) return cudaSuccess;
    if (few) {
        dim3 g1((N + 127) / 128, M, nz);
        if (c_is_f32)
            k_gemv_f64<float><<<g1, 128, 0, st>>>(N, koff, A, lda, B, ldb, (float*)C, ldc, zstride_c);
        else
            k_gemv_f64<double><<<g1, 128, 0, st>>>(N, koff, A, lda, B, ldb, (double*)C, ldc, zstride_c);
        return cudaGetLastError();
    }
    if (b_nonneg) {
        dim3 grid((N + 31) / 32, (M + 63) / 64, nz);
        if (c_is_f32)
            k_gemm_i64<float><<<grid, 256, 0, st>>>(M, N, koff, A, lda, B, ldb, (float*)C, ldc, zstride_c);
        else
            k_gemm_i64<double><<<grid, 256, 0, st>>>(M, N, koff, A, lda, B, ldb, (double*)C, ldc, zstride_c);
        return cudaGetLastError();
    }
    dim3 grid((N + 63) / 64, (M + 63) / 64, nz);
    if (c_is_f32)
        k_gemm_f64<float><<<grid, 256, 0, st>>>(M, N, koff, A, lda, B, ldb, (float*)C, ldc, zstride_c);
    else
        k_gemm_f64<double><<<grid, 256, 0, st>>>(M, N, koff, A, lda, B, ldb, (double*)C, ldc, zstride_c);
    return cudaGetLastError();
}

}  // namespace heat
