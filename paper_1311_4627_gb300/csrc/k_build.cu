// Per-solve kernels before the recursion: field tables (log-log slopes of u) and the matrix
// build (B band, Eq. bmatrix telescoped, intra-bin terms; or the point rule of Eq. heating
// with the suffix sums of Eq. brecurrence), as lane-per-cell kernels (warp = grain x 32 cells)
// and element-parallel kernels for solves of few cells.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "seg64.cuh"

namespace heat {

// ---------------------------------------------------------------------------
// k_field: transpose the chunk's fields to [N][Cc] and form the log-log slope of
// u on each segment.  ua_n = u_n where both ends of segment n are > 0 (else 0),
// su_n = ln(u_{n+1}/u_n) / ln(lambda_{n+1}/lambda_n) (else 0); ua, su = 0 at n = N-1
// and for padding cells.  Negative or non-finite input sets kStatBadInput.
// Block (32, 8) handles 32 wavelengths x 32 cells.
template <typename TU, typename TO>
__global__ void k_field(int N, const double* __restrict__ dln, const TU* __restrict__ u, long long cell0, int cells,
                        int Cc, TO* __restrict__ ua, TO* __restrict__ su, int* status) {
    __shared__ TO t_ua[32][33];
    __shared__ TO t_su[32][33];
    int n0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
    int tx = threadIdx.x, ty = threadIdx.y;
    int bad = 0;
    for (int k = 0; k < 4; ++k) {
        int c = c0 + ty + 8 * k, n = n0 + tx;
        TO a = 0, s = 0;
        if (c < cells && n < N) {
            const TU* row = u + (size_t)(cell0 + c) * N;
            double un = (double)row[n];
            if (!(un >= 0.0 && un < INFINITY)) bad = 1;
            if (n < N - 1) {
                double un1 = (double)row[n + 1];
                if (sizeof(TO) == 8) {
                    if (un > 0.0 && un1 > 0.0 && un1 < INFINITY && un < INFINITY) {
                        a = (TO)un;
                        s = (TO)(log(un1 / un) / dln[n]);
                    }
                } else {
                    float fa = (float)un, fb = (float)un1;
                    if (fa > 0.0f && fb > 0.0f && fa < INFINITY && fb < INFINITY) {
                        a = (TO)fa;
                        s = (TO)(logf(fb / fa) / (float)dln[n]);
                    }
                }
            }
        }
        t_ua[ty + 8 * k][tx] = a;
        t_su[ty + 8 * k][tx] = s;
    }
    __syncthreads();
    for (int k = 0; k < 4; ++k) {
        int n = n0 + ty + 8 * k, c = c0 + tx;
        if (n < N && c < Cc) {
            if (sizeof(TO) == 8) {
                ua[(size_t)n * Cc + c] = t_ua[tx][ty + 8 * k];
                su[(size_t)n * Cc + c] = t_su[tx][ty + 8 * k];
            } else {  // FP32 build: interleaved (u, slope) pairs, one 8-byte load per element
                float2 v = make_float2((float)t_ua[tx][ty + 8 * k], (float)t_su[tx][ty + 8 * k]);
                ((float2*)ua)[(size_t)n * Cc + c] = v;
            }
        }
    }
    if (bad) atomicOr(status, kStatBadInput);
}

// ---------------------------------------------------------------------------
// k_build: the matrix-build kernel.  One warp per task (grain x 32 cells), one lane
// per cell.  With Omega = u C on the log-log interpolant (Eq. interpolation), slope
// s_n and q = s_n + p + 1 on segment n:
//   segment integral   int Omega lambda^p = Omega_n lambda_n^{p+1} dln_n E1(q dln_n)
//   photon prefix      Phi_n = (1/h) sum_{m<n} int_m Omega lambda       (cumulative sum: FP64 in
//                      the FP64 build, compensated FP32 in the FP32 build)
//   band element       B_fj = Phi(lambda_fj) = Phi_n + (Omega_n lambda_n^2/h) t E1(q t)
//                      (Eq. bmatrix telescoped: the bins' wavelength ranges tile [0, lambda_fj])
//   intra-bin term     W_j = c int_{hc/(Elo_{j+1}-E_j)}^{lambda_{N-1}} Omega, added to the diagonal
//                      element: B_{j+1,j} += W_j/(E_{j+1}-E_j)
//   absorbed power     c int Omega over the grid
// The segments are walked in order; every band element whose transition wavelength
// falls in the current segment (the grain's pattern list) is written to the band
// storage Bb, so the recursion streams B instead of gathering tables.
template <int BUILD, bool PF = false>
__device__ __forceinline__ void build_task(const GrainDev& gd, const ChunkDev& ch, int task, int lane) {
    const int N = gd.N, Cc = ch.Cc;
    const int2 tk = (ch.btasks ? ch.btasks : ch.tasks)[task];
    int g = tk.x, grp = tk.y;
    int off = gd.bin_off[g];
    int cc = grp * 32 + lane;
    size_t bb = (size_t)grp * gd.band_total * 32 + lane;  // + e * 32
    const int* sp = gd.seg_ptr + (size_t)g * (N + 1);
    const SoftF64* soft = gd.soft;
    int p = gd.soft_off[g], p1 = gd.soft_off[g + 1];
    double Phi = 0.0;

    if (BUILD == 0) {
        const double* sC = gd.sC + (size_t)g * N;
        for (int n = 0; n < N - 1; ++n) {
            const double ua = ch.ua64[(size_t)n * Cc + cc], su = ch.su64[(size_t)n * Cc + cc];
            const SegF64 sg(gd, g, n, ua, su);
            for (int k = sp[n]; k < sp[n + 1]; ++k) {
                const PatF64 pt = gd.pat64[k];
                ch.Bb64[bb + (size_t)pt.e * 32] = sg.element(Phi, pt.t, pt.tau);
            }
            Phi = add_segment(Phi, sg.a, sg.q1, gd.dln[n]);
        }
        for (int k = sp[N - 1]; k < sp[N]; ++k) ch.Bb64[bb + (size_t)gd.pat64[k].e * 32] = Phi;

        // intra-bin terms go into the diagonal elements (j+1, j) of the band
        auto put64 = [&](const SoftF64& sf, double v) {
            size_t ix = bb + (size_t)sf.e_diag * 32;
            ch.Bb64[ix] = sf.diag_in_band ? __dadd_rn(ch.Bb64[ix], v) : v;
        };
        while (p < p1 && soft[p].n == N - 1) ++p;  // no photon is too soft: nothing to add
        double Psi = 0.0;  // int Omega from lambda_{n+1} to lambda_{N-1}
        for (int n = N - 2; n >= 0; --n) {
            const double ua = ch.ua64[(size_t)n * Cc + cc], su = ch.su64[(size_t)n * Cc + cc];
            while (p < p1 && soft[p].n == n) {
                const SoftF64 sf = soft[p];
                put64(sf, soft_term(gd, g, n, ua, su, sf.t, sf.tau, Psi, gd.invdE[off + sf.j]));
                ++p;
            }
            Psi = add_segment(Psi, ua * gd.ce64[(size_t)g * N + n], su + sC[n] + 1.0, gd.dln[n]);
        }
        for (; p < p1; ++p) put64(soft[p], soft_end(Psi, gd.invdE[off + soft[p].j]));
        if (ch.pabs) ch.pabs[(size_t)cc * gd.G + g] = kC * Psi;
    } else {
        const float* ca = gd.ca32 + (size_t)g * N;
        const float* ce = gd.ce32 + (size_t)g * N;
        const float* sC = gd.sC32 + (size_t)g * N;
        const float2* uasu = (const float2*)ch.ua32;
        float* Bb = ch.Bb32 + bb;
        float2 us_next = uasu[cc];
        Sum32 Phi32;  // the photon prefix, compensated in FP32
        for (int n = 0; n < N - 1; ++n) {
            float2 us = us_next;
            if (n + 1 < N - 1) us_next = uasu[(size_t)(n + 1) * Cc + cc];  // one segment ahead
            float ua = us.x, su = us.y;
            float phi = Phi32.val();
            int k = sp[n], k1 = sp[n + 1];
            // PF: L1 prefetch of the pattern line 32 entries past this segment (about three segments
            // ahead; the table is padded for it).  Measured on the batched workload (1024
            // wavelengths), A/B in one run: none 4.10 ms, 8 entries 3.93, 16 3.92, 32 3.87, 64 3.88,
            // 128 3.90, two lines 3.94; on the 2048-wavelength emissivity-heavy one it is slower
            // (70.5 -> 87.1 ms), so the host picks the variant per grid (heat_opts.build_prefetch)
            if (PF) asm volatile("prefetch.global.L1 [%0];" ::"l"(gd.pat32 + k1 + 32));
            // every element's argument is z = q t with t in [0, dln]: when |q| dln <= 1/4 the
            // short series serves the whole segment.  The test is per lane (per cell), so a
            // cell's values do not depend on the cells sharing its warp; lanes normally agree
            if (short_series(su, sC[n], gd.dln32[n])) {
                for (; k + 2 <= k1; k += 2) {
                    PatF32 a0 = gd.pat32[k], a1 = gd.pat32[k + 1];
                    __stcs(Bb + (size_t)a0.e * 32, fmaf(ua * a0.cat, e1f_small(fmaf(su, a0.t, a0.zt)), phi));
                    __stcs(Bb + (size_t)a1.e * 32, fmaf(ua * a1.cat, e1f_small(fmaf(su, a1.t, a1.zt)), phi));
                }
                if (k < k1) {
                    PatF32 a0 = gd.pat32[k];
                    __stcs(Bb + (size_t)a0.e * 32, fmaf(ua * a0.cat, e1f_small(fmaf(su, a0.t, a0.zt)), phi));
                }
            } else {
                for (; k + 2 <= k1; k += 2) {
                    PatF32 a0 = gd.pat32[k], a1 = gd.pat32[k + 1];
                    __stcs(Bb + (size_t)a0.e * 32, fmaf(ua * a0.cat, e1f(fmaf(su, a0.t, a0.zt)), phi));
                    __stcs(Bb + (size_t)a1.e * 32, fmaf(ua * a1.cat, e1f(fmaf(su, a1.t, a1.zt)), phi));
                }
                if (k < k1) {
                    PatF32 a0 = gd.pat32[k];
                    __stcs(Bb + (size_t)a0.e * 32, fmaf(ua * a0.cat, e1f(fmaf(su, a0.t, a0.zt)), phi));
                }
            }
            float a = ua * ca[n];
            if (a > 0.0f) {
                float dl = gd.dln32[n];
                Phi32.add(a * dl * e1f((su + sC[n] + 2.0f) * dl));
            }
        }
        float phi_end = Phi32.val();
        for (int k = sp[N - 1]; k < sp[N]; ++k) Bb[gd.pat32[k].e * 32] = phi_end;

        auto put32 = [&](const SoftF64& sf, float v) {
            float* q = Bb + (size_t)sf.e_diag * 32;
            *q = (sf.diag_in_band ? *q : 0.0f) + v;
        };
        while (p < p1 && soft[p].n == N - 1) {
            put32(soft[p], 0.0f);
            ++p;
        }
        Sum32 Psi32;  // c int Omega from lambda_{n+1} to lambda_{N-1} (compensated FP32 sum)
        us_next = uasu[(size_t)(N - 2) * Cc + cc];
        for (int n = N - 2; n >= 0; --n) {
            float2 us = us_next;
            if (n > 0) us_next = uasu[(size_t)(n - 1) * Cc + cc];
            float ua = us.x, su = us.y;
            float b = ua * ce[n];
            float q0 = su + sC[n] + 1.0f;
            float dl = gd.dln32[n];
            while (p < p1 && soft[p].n == n) {
                SoftF64 sf = soft[p];
                float part = 0.0f;
                if (b > 0.0f) {
                    float ts = (float)sf.t;
                    float L = dl - ts;
                    part = b * __expf(q0 * ts) * L * e1f(q0 * L);
                }
                put32(sf, (part + Psi32.val()) * gd.invdE32[off + sf.j]);
                ++p;
            }
            if (b > 0.0f) Psi32.add(b * dl * e1f(q0 * dl));
        }
        float psi_end = Psi32.val();
        for (; p < p1; ++p) put32(soft[p], psi_end * gd.invdE32[off + soft[p].j]);
        if (ch.pabs) ch.pabs[(size_t)cc * gd.G + g] = Psi32.wide();
    }
}

// One warp per task, in the build's task order.
template <int BUILD, bool PF = false>
__global__ void __launch_bounds__(128) k_build(GrainDev gd, ChunkDev ch) {
    const int task = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (task < ch.n_tasks) build_task<BUILD, PF>(gd, ch, task, threadIdx.x & 31);
}

// ---------------------------------------------------------------------------
// The build in two passes.  One walk per (grain, 32-cell group) leaves the device to the tasks
// with the most elements once the others are done (on average 19 of the 48 warps an SM holds were
// active), and takes as long as its longest task however few the cells.  So:
//   k_prefix  the walks alone, one warp per (grain, group, direction): forward, Phi at every
//             wavelength node into phi[g][n][cell]; backward, the intra-bin terms, parked in the
//             diagonal elements' places of the band, and the absorbed power;
//   k_elem    the band elements in pieces of kPieceEntries pattern entries: any number of warps,
//             all alike.  A diagonal element adds the term it finds in its place.
// The sums run in k_build's order and every expression is k_build's, so B is bit for bit the same.
// Measured (FP32 build, one walk -> two passes): 4096 cells x 64 grains x 1024 wavelengths 3.88 -> 3.10 ms
// (elements 2.0 ms, 5.5 TB/s, what the band's 10.2 GB of stores leaves; walks 1.1 ms); 1003 x 37 x 771
// 2.95 -> 0.75 ms; 4096 x 32 x 2048 with 512 bins 19.9 -> 3.4 ms; 4096 x 80 x 1024 with 512 bins 37.6 -> 11.0 ms.
// The prefix table costs 4 (8) bytes per grain, wavelength and cell; without room for it the one walk runs.
// FP64 walks: a warp per (direction, group, grain).  Backward, a diagonal element's place takes Psi, from which
// the element pass makes the intra-bin term.
__global__ void __launch_bounds__(128) k_prefix64(GrainDev gd, ChunkDev ch) {
    const int N = gd.N, Cc = ch.Cc, lane = threadIdx.x & 31;
    // the grains of one group and direction in turn, so that the warps of a block read the same fields
    long long w = (long long)blockIdx.x * 4 + (threadIdx.x >> 5);
    const int g = (int)(w % gd.G);
    w /= gd.G;
    const int grp = (int)(w % ch.NG), back = (int)(w / ch.NG);
    if (back > 1) return;
    const int off = gd.bin_off[g], cc = grp * 32 + lane;
    const size_t bb = (size_t)grp * gd.band_total * 32 + lane;
    constexpr int U = 2;  // segments whose series run side by side
    const double* __restrict__ cf = (back ? gd.ce64 : gd.ca64) + (size_t)g * N;
    const double* __restrict__ sC = gd.sC + (size_t)g * N;
    const double* __restrict__ ua = ch.ua64 + cc;
    const double* __restrict__ su = ch.su64 + cc;
    double* phi = back ? nullptr : ch.phi64 + (size_t)g * N * Cc + cc;
    const SoftF64* __restrict__ soft = gd.soft;
    int p = 0, p1 = 0, pn = -2;
    if (back) {
        p = gd.soft_off[g];
        p1 = gd.soft_off[g + 1];
        while (p < p1 && soft[p].n == N - 1) ++p;  // no photon is too soft: nothing to add
        pn = p < p1 ? soft[p].n : -2;
    }
    double sum = 0.0;
    for (int i0 = 0; i0 < N - 1; i0 += U) {
        double m[U], e[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int i = min(i0 + k, N - 2), n = back ? N - 2 - i : i;
            const double v = ua[(size_t)n * Cc] * cf[n], q = su[(size_t)n * Cc] + sC[n] + (back ? 1.0 : 2.0);
            const double dl = gd.dln[n];
            m[k] = v > 0.0 ? v * dl : 0.0;
            e[k] = v > 0.0 ? e1_of(q * dl) : 0.0;
        }
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int i = i0 + k, n = back ? N - 2 - i : i;
            if (i >= N - 1) break;
            if (!back) phi[(size_t)n * Cc] = sum;
            while (pn == n) {
                ch.Bb64[bb + (size_t)soft[p].e_diag * 32] = sum;
                ++p;
                pn = p < p1 ? soft[p].n : -2;
            }
            sum = fma(m[k], e[k], sum);
        }
    }
    if (!back) {
        phi[(size_t)(N - 1) * Cc] = sum;
        return;
    }
    for (; p < p1; ++p)  // no photon on the grid reaches the next bin: all absorbed power counts
        ch.Bb64[bb + (size_t)soft[p].e_diag * 32] = soft_end(sum, gd.invdE[off + soft[p].j]);
    if (ch.pabs) ch.pabs[(size_t)cc * gd.G + g] = kC * sum;
}

// FP32 walks: a warp takes two grains, one direction, one group of cells.  The two grains share the
// field loads and run through the packed FP32 instructions (each half rounds as the scalar one).
// Bound by issue and by the few warps a walk has (2048 cells: 44 % of the issue slots, 76
// instructions per segment and pair); four grains a warp, or scalar instructions with one grain, took
// 1.06 ms at 2048 cells against 0.62.
__global__ void __launch_bounds__(128) k_prefix32(GrainDev gd, ChunkDev ch) {
    const int N = gd.N, Cc = ch.Cc, lane = threadIdx.x & 31, GP = (gd.G + 1) / 2;
    // the groups of one pair of grains in turn: a block's warps read the same segment table
    long long w = (long long)blockIdx.x * 4 + (threadIdx.x >> 5);
    const int grp = (int)(w % ch.NG);
    w /= ch.NG;
    const int q = (int)(w % GP), back = (int)(w / GP), g0 = 2 * q;
    if (back > 1) return;
    const bool two = g0 + 1 < gd.G;
    const int cc = grp * 32 + lane;
    const int last = N - 2, dir = back ? -1 : 1;
    const ptrdiff_t cstep = (ptrdiff_t)Cc * dir;
    // the next segment to load, in the walk's direction
    const float2* us_p = (const float2*)ch.ua32 + cc + (back ? (size_t)last * Cc : 0);
    const float4* tab = gd.seg32 + ((size_t)back * GP + q) * N + (back ? last : 0);
    const float* dln = gd.dln32 + (back ? last : 0);
    constexpr int U = 4;  // segments loaded together, a batch ahead of their use
    float2 us[U], us_n[U];
    float4 c[U], c_n[U];
    float dl[U], dl_n[U];
    Sum32x2 S;
    auto load = [&](int i0, float2(&u)[U], float4(&t)[U], float(&d)[U]) {  // steps i0 .. i0 + U - 1
#pragma unroll
        for (int k = 0; k < U; ++k)
            if (i0 + k <= last) {
                u[k] = us_p[k * cstep];
                t[k] = __ldg(tab + k * dir);
                d[k] = __ldg(dln + k * dir);
            }
        us_p += U * cstep;
        tab += U * dir;
        dln += U * dir;
    };
    // a step's increments v dl E1((su + sC + p + 1) dl) of both grains (0 where v is 0)
    auto increment = [&](F2 v, F2 qv, F2 d2) {
        const F2 z = mul2(qv, d2), m = mul2(v, d2);
        if (fmaxf(fabsf(lo(z)), fabsf(hi(z))) < 0.5f) return mul2(m, e1f_series2(z));
        return f2(lo(v) > 0.0f ? lo(m) * e1f(lo(z)) : 0.0f, hi(v) > 0.0f ? hi(m) * e1f(hi(z)) : 0.0f);
    };
    load(0, us, c, dl);
    if (!back) {
        float* phi0 = ch.phi32 + (size_t)g0 * N * Cc + cc;
        float* phi1 = two ? phi0 + (size_t)N * Cc : phi0;
        for (int n0 = 0; n0 < N - 1; n0 += U) {
            load(n0 + U, us_n, c_n, dl_n);
#pragma unroll
            for (int k = 0; k < U; ++k) {
                if (n0 + k > last) break;
                const F2 v = S.val();
                if (two) *phi1 = hi(v);
                *phi0 = lo(v);
                phi0 += Cc;
                phi1 += Cc;
                const F2 a = mul2(f2(us[k].x), f2(c[k].x, c[k].y));
                S.add(increment(a, add2(add2(f2(us[k].y), f2(c[k].z, c[k].w)), f2(2.0f)), f2(dl[k])));
            }
#pragma unroll
            for (int k = 0; k < U; ++k) us[k] = us_n[k], c[k] = c_n[k], dl[k] = dl_n[k];
        }
        if (two) *phi1 = hi(S.val());
        *phi0 = lo(S.val());
        return;
    }
    float* Bb = ch.Bb32 + (size_t)grp * gd.band_total * 32 + lane;
    int p[2] = {0, 0}, p1[2] = {0, 0};
    int4 sf[2] = {}, sf_n[2] = {};  // each grain's next two soft-photon records (loaded a record ahead of the test)
    auto next = [&](int i) {
        sf[i] = sf_n[i];
        sf_n[i] = __ldg(gd.soft32 + min(p[i] + 1, p1[i]));
        if (p[i] >= p1[i]) sf[i].x = -2;
    };
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int g = min(g0 + i, gd.G - 1);
        p1[i] = gd.soft_off[g + 1];
        p[i] = g0 + i < gd.G ? gd.soft_off[g] : p1[i];
        while (p[i] < p1[i] && gd.soft32[p[i]].x == N - 1) ++p[i];  // no photon is too soft: nothing to add
        sf_n[i] = __ldg(gd.soft32 + p[i]);
        next(i);
    }
    for (int i0 = 0; i0 < N - 1; i0 += U) {
        load(i0 + U, us_n, c_n, dl_n);
#pragma unroll
        for (int k = 0; k < U; ++k) {
            if (i0 + k > last) break;
            const int n = last - i0 - k;
            const F2 b = mul2(f2(us[k].x), f2(c[k].x, c[k].y));
            const F2 q0 = add2(add2(f2(us[k].y), f2(c[k].z, c[k].w)), f2(1.0f));
#pragma unroll
            for (int i = 0; i < 2; ++i)
                while (sf[i].x == n) {
                    const int4 r = sf[i];
                    ++p[i];
                    next(i);
                    const float bi = i ? hi(b) : lo(b), qi = i ? hi(q0) : lo(q0);
                    float part = 0.0f;
                    if (bi > 0.0f) {
                        const float ts = __int_as_float(r.z), L = dl[k] - ts;
                        part = bi * __expf(qi * ts) * L * e1f(qi * L);
                    }
                    const float psi = i ? hi(S.val()) : lo(S.val());
                    Bb[(size_t)r.y * 32] = __fmul_rn(__fadd_rn(part, psi), __int_as_float(r.w));
                }
            S.add(increment(b, q0, f2(dl[k])));
        }
#pragma unroll
        for (int k = 0; k < U; ++k) us[k] = us_n[k], c[k] = c_n[k], dl[k] = dl_n[k];
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        if (g0 + i >= gd.G) break;
        const float psi_end = i ? hi(S.val()) : lo(S.val());
        for (; p[i] < p1[i]; ++p[i]) {  // no photon on the grid reaches the next bin: all absorbed power counts
            const int4 r = __ldg(gd.soft32 + p[i]);
            Bb[(size_t)r.y * 32] = __fmul_rn(psi_end, __int_as_float(r.w));
        }
        if (ch.pabs)
            ch.pabs[(size_t)cc * gd.G + g0 + i] =
                i ? (double)hi(S.s) + (double)hi(S.c) : (double)lo(S.s) + (double)lo(S.c);
    }
}

// One piece of a grain's pattern entries for up to 8 warps' cells.  The piece's entries and segment
// records are staged in shared memory, where all warps read them as broadcasts; what a warp loads
// from memory is its cells' prefix and field values, a segment ahead.
// FP64: a warp per group of 32 cells, lane = cell.  Bound by the integer pipes and issue (61 % of the slots, 63
// instructions an element; the FP64 unit does two of them); 512 cells x 64 grains x 1024 wavelengths, walks
// included: 18.5 ms with the series in FP64 and one walk per task, 3.8 ms (walks 1.3, elements 2.5).
__global__ void __launch_bounds__(256) k_elem64(GrainDev gd, ChunkDev ch, int gblocks) {
    __shared__ __align__(8) PatF64 pat[kPieceEntries];
    __shared__ __align__(16) int4 seg[kPieceEntries];
    const int piece = blockIdx.x / gblocks;
    const int4 pc = gd.pieces[2 * piece], ps = gd.pieces[2 * piece + 1];
    const int N = gd.N, Cc = ch.Cc, g = pc.x, ne = pc.z - pc.y, ns = ps.y - ps.x;
    for (int i = threadIdx.x; i < 3 * ne; i += blockDim.x) ((int2*)pat)[i] = __ldg((const int2*)(gd.pat64 + pc.y) + i);
    for (int i = threadIdx.x; i < ns; i += blockDim.x) seg[i] = __ldg(gd.pseg + ps.x + i);
    __syncthreads();
    const int grp = (blockIdx.x % gblocks) * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (grp >= ch.NG) return;
    const int cc = grp * 32 + lane;
    int k = 0;
    const double* __restrict__ phi = ch.phi64 + (size_t)g * N * Cc + cc;
    const double* __restrict__ uap = ch.ua64 + cc;
    const double* __restrict__ sup = ch.su64 + cc;
    double* Bb = ch.Bb64 + (size_t)grp * gd.band_total * 32 + lane;
    for (int s = 0; s < ns; ++s) {
        const int4 r = seg[s];
        const int n = r.x;
        const double Phi = phi[(size_t)n * Cc];
        if (n == N - 1) {  // at or beyond the last node: the whole grid's prefix
            for (; k < r.z; ++k) __stcs(Bb + (size_t)pat[k].e * 32, Phi);
            break;
        }
        const double ua = uap[(size_t)n * Cc], su = sup[(size_t)n * Cc];
        const SegF64 sg(gd, g, n, ua, su);
        for (; k < r.y; ++k) __stcs(Bb + (size_t)pat[k].e * 32, sg.element(Phi, pat[k].t, pat[k].tau));
        for (; k < r.z; ++k) {  // diagonal elements: plus the intra-bin term, from the Psi in their place
            double* q = Bb + (size_t)pat[k].e * 32;
            const double v = soft_term(gd, g, n, ua, su, pat[k].t, pat[k].tau, *q, gd.invdE[pat[k].j]);
            __stcs(q, __dadd_rn(sg.element(Phi, pat[k].t, pat[k].tau), v));
        }
    }
}

// FP32: a warp per two groups (64 cells), lane = a cell of each, the two in the halves of the packed
// FP32 instructions: an entry's constants, its address and every operation serve both.
__global__ void __launch_bounds__(256) k_elem32(GrainDev gd, ChunkDev ch, int gblocks) {
    __shared__ __align__(16) PatF32 pat[kPieceEntries];
    __shared__ __align__(16) int4 seg[kPieceEntries];
    __shared__ float2 sq[kPieceEntries];  // (sC, dln) of the segments
    const int piece = blockIdx.x / gblocks;
    const int4 pc = gd.pieces[2 * piece], ps = gd.pieces[2 * piece + 1];
    const int N = gd.N, Cc = ch.Cc, g = pc.x, ne = pc.z - pc.y, ns = ps.y - ps.x;
    for (int i = threadIdx.x; i < ne; i += blockDim.x) ((int4*)pat)[i] = __ldg((const int4*)(gd.pat32 + pc.y) + i);
    for (int i = threadIdx.x; i < ns; i += blockDim.x) {
        const int4 r = __ldg(gd.pseg + ps.x + i);
        seg[i] = r;
        sq[i] = r.x < N - 1 ? make_float2(gd.sC32[(size_t)g * N + r.x], gd.dln32[r.x]) : make_float2(0.0f, 0.0f);
    }
    __syncthreads();
    const int grp = 2 * ((blockIdx.x % gblocks) * (blockDim.x >> 5) + (threadIdx.x >> 5)), lane = threadIdx.x & 31;
    if (grp >= ch.NG) return;
    const bool two = grp + 1 < ch.NG;  // else the second half repeats the first and is not stored
    const int cc = grp * 32 + lane, c1 = two ? 32 : 0;
    const float* __restrict__ phis = ch.phi32 + (size_t)g * N * Cc + cc;
    const float2* __restrict__ uasu = (const float2*)ch.ua32 + cc;
    float* B0 = ch.Bb32 + (size_t)grp * gd.band_total * 32 + lane;
    float* B1 = B0 + (two ? (size_t)gd.band_total * 32 : 0);
    int k = 0;
    int4 r = seg[0];
    float2 ph, ua, ub;  // the next segment's prefix and (u, slope) of both cells
    auto load = [&] {
        const size_t n = (size_t)r.x * Cc;
        ph = make_float2(phis[n], phis[n + c1]);
        ua = uasu[n];
        ub = uasu[n + c1];
    };
    load();
    for (int s = 0; s < ns; ++s) {
        const int n = r.x, kd = r.y, ke = r.z;
        const F2 phi = f2(ph.x, ph.y), u = f2(ua.x, ub.x), su = f2(ua.y, ub.y);
        const float2 sc = sq[s];
        if (s + 1 < ns) {
            r = seg[s + 1];
            load();
        }
        if (n == N - 1) {  // at or beyond the last node: the whole grid's prefix
            for (; k < ke; ++k) {
                const size_t o = (size_t)pat[k].e * 32;
                __stcs(B0 + o, lo(phi));
                if (two) __stcs(B1 + o, hi(phi));
            }
            break;
        }
        // the series is chosen per cell (lanes and halves normally agree), so that a cell's values do not
        // depend on the cells beside it
        const bool s0 = short_series(lo(su), sc.x, sc.y), s1 = short_series(hi(su), sc.x, sc.y);
        auto run = [&](auto e1) {
            auto elem = [&](const PatF32& a) {
                return fma2(mul2(u, f2(a.cat)), e1(fma2(su, f2(a.t), f2(a.zt))), phi);
            };
#pragma unroll 4
            for (; k < kd; ++k) {
                const PatF32 a = pat[k];
                const F2 b = elem(a);
                const size_t o = (size_t)a.e * 32;
                __stcs(B0 + o, lo(b));
                if (two) __stcs(B1 + o, hi(b));
            }
            for (; k < ke; ++k) {  // diagonal elements: plus the intra-bin term parked in their place
                const PatF32 a = pat[k];
                const size_t o = (size_t)a.e * 32;
                const F2 b = add2(elem(a), f2(B0[o], B1[o]));
                __stcs(B0 + o, lo(b));
                if (two) __stcs(B1 + o, hi(b));
            }
        };
        if (s0 && s1)
            run([](F2 z) { return e1f_small2(z); });
        else
            run([&](F2 z) { return f2(s0 ? e1f_small(lo(z)) : e1f(lo(z)), s1 ? e1f_small(hi(z)) : e1f(hi(z))); });
        k = ke;
    }
}

// ---------------------------------------------------------------------------
// Element-parallel build for solves of few cells (ChunkDev::small): the same quantities as
// k_build with the same expressions.  FP32: the cumulative sums run in the same order (one
// thread), so B is bit-identical.  FP64: a warp scan, so B differs in the last bits.

// Blocks per (cell, grain): S parts (256 threads each, dynamic shared memory 2 N doubles).
// Every part forms the segment increments and the cumulative sums; part q writes the
// elements of a run of segments, cut so that the parts have about as many elements each, and the
// intra-bin terms whose diagonal element it wrote: the diagonal (j+1, j) and bin j's soft-photon
// edge are the same wavelength, hc/(Elo_{j+1} - E_j), so both fall in segment sf.n (sf.n < 0: the
// diagonal is not in the band, part 0).  Few spectra (a single cell) then spread over many SMs.
// The sums are the serial part: FP32, one thread in the lane-per-cell kernel's order (its bits), on FP32 values
// throughout (a conversion to or from FP64 takes the FP64 unit 64 cycles); FP64, a warp, a run of segments a lane
// and a scan over the lanes.  The elements take a thread each.  Against a warp per segment and FP64 sums on one thread:
// 5 cells x 64 grains x 1024 wavelengths (FP32) 216 -> 119 us, single cell (FP64) 36 -> 15 us.  With the parts cut as
// segments n = q (mod S), each part looking through all entries for its own: 130 and 23 us, and a cell of 8 grains of 900
// bins, all reaching each other, 296 -> 805 us where this takes 258.
template <int BUILD>
__global__ void __launch_bounds__(256, BUILD ? 6 : 5) k_build_small(GrainDev gd, ChunkDev ch, int S) {
    using Real = typename std::conditional<BUILD == 0, double, float>::type;
    extern __shared__ double sm[];
    Real* sPhi = (Real*)sm;     // [N]: Phi before segment n (exclusive prefix)
    Real* sPsi = sPhi + gd.N;   // [N]: Psi after the segments above n (exclusive suffix)
    __shared__ Real sPhiEnd;
    __shared__ int s_seg[2];
    __shared__ double sPsiTot;
    __shared__ float sPsiEnd32;  // FP32 build: the FP32 value of the compensated total
    const int N = gd.N, Cc = ch.Cc;
    const int spec = blockIdx.x / S, part = blockIdx.x % S;
    const int cell = spec / gd.G, g = spec % gd.G;
    if (cell >= ch.cells) return;
    const int grp = cell >> 5, lc = cell & 31;
    const int off = gd.bin_off[g];
    const size_t bb = (size_t)grp * gd.band_total * 32 + lc;
    const int* sp = gd.seg_ptr + (size_t)g * (N + 1);
    const int tid = threadIdx.x, lane = tid & 31;
    const float2* uasu = (const float2*)ch.ua32;
    // 1. segment increments, in parallel
    for (int n = tid; n < N - 1; n += blockDim.x) {
        const size_t gn = (size_t)g * N + n;
        Real dphi = 0, dpsi = 0;
        if (BUILD == 0) {
            const double ua = ch.ua64[(size_t)n * Cc + cell], su = ch.su64[(size_t)n * Cc + cell];
            const double dl = gd.dln[n];
            dphi = add_segment(0.0, ua * gd.ca64[gn], su + gd.sC[gn] + 2.0, dl);
            dpsi = add_segment(0.0, ua * gd.ce64[gn], su + gd.sC[gn] + 1.0, dl);
        } else {
            const float2 us = uasu[(size_t)n * Cc + cell];
            const float ua = us.x, su = us.y;
            const float sc = gd.sC32[gn], dl = gd.dln32[n];
            const float a = ua * gd.ca32[gn];
            if (a > 0.0f) dphi = a * dl * e1f((su + sc + 2.0f) * dl);
            const float b = ua * gd.ce32[gn];
            if (b > 0.0f) dpsi = b * dl * e1f((su + sc + 1.0f) * dl);
        }
        sPhi[n] = dphi;
        sPsi[n] = dpsi;
    }
    __syncthreads();
    if (tid >= 64 && tid < 66) {  // beside the sums: the first segment whose entries begin at or after q / S of all
        const int q = part + tid - 64;
        int lo = 0, hi = N;
        while (lo < hi && q < S) {
            const int mid = (lo + hi) >> 1;
            if ((long long)(sp[mid] - sp[0]) * S >= (long long)q * (sp[N] - sp[0])) hi = mid; else lo = mid + 1;
        }
        s_seg[tid - 64] = q == 0 ? 0 : q < S ? lo : N;
    }
    // 2. the cumulative sums
    if constexpr (BUILD == 0) {
        if (tid < 64) {  // warp 0 upward over sPhi, warp 1 downward over sPsi
            const bool down = tid >= 32;
            Real* v = down ? sPsi : sPhi;
            const int per = (N - 1 + 31) / 32, i0 = min(lane * per, N - 1), i1 = min(i0 + per, N - 1);
            double run = 0.0;
            for (int i = i0; i < i1; ++i) run += v[down ? N - 2 - i : i];
            double incl = run;
            for (int o = 1; o < 32; o <<= 1) {
                const double t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            double before = __shfl_up_sync(0xffffffffu, incl, 1);
            if (lane == 0) before = 0.0;
            for (int i = i0; i < i1; ++i) {
                const int n = down ? N - 2 - i : i;
                const double d = v[n];
                v[n] = before;
                before += d;
            }
            const double tot = __shfl_sync(0xffffffffu, incl, 31);
            if (lane == 0) {
                if (down)
                    sPsiTot = tot;
                else
                    sPhiEnd = tot;
            }
        }
    } else if (tid == 0 || tid == 32) {
        // the increments are read eight at a time ahead of the sums, so that no shared-memory load latency sits on
        // the sums' dependent chain
        constexpr int R = 8;
        const bool down = tid == 32;
        Real* v = down ? sPsi : sPhi;
        Sum32 sum;
        for (int i0 = 0; i0 < N - 1; i0 += R) {
            float d[R];
#pragma unroll
            for (int k = 0; k < R; ++k) d[k] = i0 + k < N - 1 ? (float)v[down ? N - 2 - i0 - k : i0 + k] : 0.0f;
#pragma unroll
            for (int k = 0; k < R; ++k)
                if (i0 + k < N - 1) {
                    v[down ? N - 2 - i0 - k : i0 + k] = sum.val();
                    sum.add(d[k]);
                }
        }
        if (down) {
            sPsiTot = sum.wide();
            sPsiEnd32 = sum.val();
        } else {
            sPhiEnd = sum.val();
        }
    }
    __syncthreads();
    // 3. band elements of this part's segments [n_lo, n_hi), a thread each
    const int n_lo = s_seg[0], n_hi = s_seg[1];
    for (int k = sp[n_lo] + tid, k1 = sp[min(n_hi, N - 1)]; k < k1; k += blockDim.x) {
        const int n = BUILD ? gd.pat_seg[k] : __ldcs(gd.pat_seg + k);
        if (BUILD == 0) {
            const SegF64 s(gd, g, n, ch.ua64[(size_t)n * Cc + cell], ch.su64[(size_t)n * Cc + cell]);
            PatF64 pt;  // evict first: the recursion reads B next, which alone can fill the L2
#pragma unroll
            for (int w = 0; w < 3; ++w) ((int2*)&pt)[w] = __ldcs((const int2*)(gd.pat64 + k) + w);
            ch.Bb64[bb + (size_t)pt.e * 32] = s.element(sPhi[n], pt.t, pt.tau);
        } else {
            const float2 us = uasu[(size_t)n * Cc + cell];
            const bool sh = short_series(us.y, gd.sC32[(size_t)g * N + n], gd.dln32[n]);
            const PatF32 a0 = gd.pat32[k];
            const float z = fmaf(us.y, a0.t, a0.zt);
            ch.Bb32[bb + (size_t)a0.e * 32] = fmaf(us.x * a0.cat, sh ? e1f_small(z) : e1f(z), (float)sPhi[n]);
        }
    }
    if (n_lo <= N - 1 && N - 1 < n_hi)
        for (int k = sp[N - 1] + tid; k < sp[N]; k += blockDim.x) {
            if (BUILD == 0)
                ch.Bb64[bb + (size_t)gd.pat64[k].e * 32] = sPhiEnd;
            else
                ch.Bb32[bb + (size_t)gd.pat32[k].e * 32] = (float)sPhiEnd;
        }
    __syncthreads();  // the intra-bin terms add to diagonal elements written above (by this part)
    // 4. intra-bin terms, one per soft entry (each has its own diagonal element)
    for (int p = gd.soft_off[g] + tid; p < gd.soft_off[g + 1]; p += blockDim.x) {
        const SoftF64 sf = gd.soft[p];
        if (sf.n < 0 ? part != 0 : sf.n < n_lo || sf.n >= n_hi) continue;
        if (BUILD == 0) {
            double v = 0.0;
            if (sf.n == N - 1) {
                v = 0.0;
            } else if (sf.n >= 0) {
                v = soft_term(gd, g, sf.n, ch.ua64[(size_t)sf.n * Cc + cell], ch.su64[(size_t)sf.n * Cc + cell], sf.t, sf.tau,
                              sPsi[sf.n], gd.invdE[off + sf.j]);
            } else {
                v = soft_end(sPsiTot, gd.invdE[off + sf.j]);
            }
            const size_t ix = bb + (size_t)sf.e_diag * 32;
            ch.Bb64[ix] = (sf.diag_in_band ? ch.Bb64[ix] : 0.0) + v;
        } else {
            float v = 0.0f;
            if (sf.n == N - 1) {
                v = 0.0f;
            } else if (sf.n >= 0) {
                const float2 us = uasu[(size_t)sf.n * Cc + cell];
                const float b = us.x * gd.ce32[(size_t)g * N + sf.n];
                const float q0 = us.y + gd.sC32[(size_t)g * N + sf.n] + 1.0f;
                const float dl = gd.dln32[sf.n];
                float part = 0.0f;
                if (b > 0.0f) {
                    const float ts = (float)sf.t;
                    const float L = dl - ts;
                    part = b * __expf(q0 * ts) * L * e1f(q0 * L);
                }
                v = (part + (float)sPsi[sf.n]) * gd.invdE32[off + sf.j];
            } else {
                v = sPsiEnd32 * gd.invdE32[off + sf.j];
            }
            float* q = ch.Bb32 + bb + (size_t)sf.e_diag * 32;
            *q = (sf.diag_in_band ? *q : 0.0f) + v;
        }
    }
    if (tid == 0 && part == 0 && ch.pabs) ch.pabs[(size_t)cell * gd.G + g] = BUILD == 0 ? kC * sPsiTot : sPsiTot;
}

// ---------------------------------------------------------------------------
// Point-rule build (HEAT_HEATING_POINT; Eq. heating at the bin centres, Eq. brecurrence):
//   T_uj = Omega(lambda_uj) lambda_uj^3 dE_u / (h^2 c),  Omega(lambda) = u_n C_n e^{(su_n + sC_n) t}
// on the log-log interpolant (the slope of the product u C is the sum of the slopes), and
// B_uj = B_{u+1,j} + T_uj down each column from its last band row, in the order of the
// suffix recurrence.  Every band element is written (elements the rule leaves at zero
// carry the column's sum).  Also the absorbed power c int Omega on the grid, summed in
// k_build's order, for the energy check.
__device__ __forceinline__ void point_column(const GrainDev& gd, const ChunkDev& ch, int g, int cell, int j,
                                             double* Bb) {
    const int N = gd.N, Cc = ch.Cc;
    const double* Cact = gd.Cact + (size_t)g * N;
    const double* sC = gd.sC + (size_t)g * N;
    const int off = gd.bin_off[g];
    const int k1 = gd.pcol[off + j + 1];
    double acc = 0.0, om = 0.0, s = 0.0;
    int64_t Z = 0;
    int cls = 1, ncur = -1;
    for (int k = gd.pcol[off + j]; k < k1; ++k) {
        const PointEnt pe = gd.pent[k];
        if (pe.n >= 0) {
            if (pe.n != ncur) {  // entries move up the wavelength grid along a column
                ncur = pe.n;
                om = ch.ua64[(size_t)pe.n * Cc + cell] * Cact[pe.n];
                s = ch.su64[(size_t)pe.n * Cc + cell] + sC[pe.n];
                const double z = s * gd.dln[pe.n];
                cls = e1_class(z);
                Z = cls ? to_q60(z) : 0;
            }
            double e;  // e^{s t} = 1 + z E1(z), in fixed point where |s| dln < 1
            if (cls) {
                const int64_t z = mul_q60(Z, pe.tau);
                e = from_q60(kQ60 + mul_q60(z, e1_q60(cls, z)));
            } else {
                e = exp(s * pe.t);
            }
            acc = fma(om * pe.fac, e, acc);
        }
        __stcs(Bb + (size_t)pe.e * 32, acc);
    }
}

// c int Omega over the grid, in the order and arithmetic of the integral form's walk
__device__ __forceinline__ double absorbed_power(const GrainDev& gd, const ChunkDev& ch, int g, int cell) {
    const int N = gd.N, Cc = ch.Cc;
    const double* ce = gd.ce64 + (size_t)g * N;
    const double* sC = gd.sC + (size_t)g * N;
    double Psi = 0.0;
    for (int n = N - 2; n >= 0; --n)
        Psi = add_segment(Psi, ch.ua64[(size_t)n * Cc + cell] * ce[n], ch.su64[(size_t)n * Cc + cell] + sC[n] + 1.0,
                          gd.dln[n]);
    return kC * Psi;
}

// Lane per cell, a warp per run of columns of about kPointEntries entries (any number of warps, all alike: with a
// warp per (grain, 32 cells) 203 cells of 19 grains were 133 warps on 608 sub-partitions), then a warp per
// (grain, 32 cells) for the absorbed power.  203 cells x 19 grains x 500
// wavelengths: 17.6 ms with a warp per task and FP64 exponentials, 0.64 ms.
__global__ void __launch_bounds__(128) k_build_point(GrainDev gd, ChunkDev ch) {
    long long w = (long long)blockIdx.x * 4 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    const long long power = ch.pabs ? (long long)gd.G * ch.NG : 0;
    if (w < power) {  // the longest chains first
        const int g = (int)(w / ch.NG), cell = (int)(w % ch.NG) * 32 + lane;
        ch.pabs[(size_t)cell * gd.G + g] = absorbed_power(gd, ch, g, cell);
        return;
    }
    w -= power;
    if (w >= (long long)gd.n_cpieces * ch.NG) return;
    const int4 pc = gd.cpieces[w / ch.NG];
    const int grp = (int)(w % ch.NG), cell = grp * 32 + lane;
    double* Bb = ch.Bb64 + (size_t)grp * gd.band_total * 32 + lane;
    for (int j = pc.y; j < pc.z; ++j) point_column(gd, ch, pc.x, cell, j, Bb);
}

// Few cells: block per (cell, grain), threads over the columns (each column's sum is the
// same sequence as in k_build_point, so B is bit-identical).
__global__ void __launch_bounds__(128) k_build_point_small(GrainDev gd, ChunkDev ch) {
    const int cell = blockIdx.x / gd.G, g = blockIdx.x % gd.G;
    if (cell >= ch.cells) return;
    const int M = gd.bin_off[g + 1] - gd.bin_off[g] - 1;
    double* Bb = ch.Bb64 + (size_t)(cell >> 5) * gd.band_total * 32 + (cell & 31);
    for (int j = threadIdx.x; j < M; j += blockDim.x) point_column(gd, ch, g, cell, j, Bb);
    if (threadIdx.x == 0 && ch.pabs) ch.pabs[(size_t)cell * gd.G + g] = absorbed_power(gd, ch, g, cell);
}

cudaError_t launch_field(const GrainDev& g, const void* u, int dtype, long long cell0, const ChunkDev& ch, int build,
                         cudaStream_t st) {
    dim3 block(32, 8), grid((g.N + 31) / 32, ch.Cc / 32);
    if (build == 0) {
        if (dtype == 0)
            k_field<double, double><<<grid, block, 0, st>>>(g.N, g.dln, (const double*)u, cell0, ch.cells, ch.Cc, ch.ua64,
                                                            ch.su64, ch.status);
        else
            k_field<float, double><<<grid, block, 0, st>>>(g.N, g.dln, (const float*)u, cell0, ch.cells, ch.Cc, ch.ua64,
                                                           ch.su64, ch.status);
    } else {
        if (dtype == 0)
            k_field<double, float><<<grid, block, 0, st>>>(g.N, g.dln, (const double*)u, cell0, ch.cells, ch.Cc, ch.ua32,
                                                           ch.su32, ch.status);
        else
            k_field<float, float><<<grid, block, 0, st>>>(g.N, g.dln, (const float*)u, cell0, ch.cells, ch.Cc, ch.ua32,
                                                          ch.su32, ch.status);
    }
    return cudaGetLastError();
}

cudaError_t launch_build(const GrainDev& g, const ChunkDev& ch, int build, cudaStream_t st) {
    if (ch.point) {  // the point rule (FP64 build only; checked by the caller)
        if (build != 0) return cudaErrorInvalidValue;
        if (ch.small) {
            const unsigned blocks = (unsigned)(ch.cells * g.G);
            if (blocks) k_build_point_small<<<blocks, 128, 0, st>>>(g, ch);
        } else {
            const long long warps = (long long)ch.NG * (g.n_cpieces + (ch.pabs ? g.G : 0));
            k_build_point<<<(unsigned)((warps + 3) / 4), 128, 0, st>>>(g, ch);
        }
        return cudaGetLastError();
    }
    if (ch.small) {
        const size_t smem = (build == 0 ? sizeof(double) : sizeof(float)) * 2 * (size_t)g.N;
        const long long spectra = (long long)ch.cells * g.G;
        if (spectra == 0) return cudaSuccess;
        // parts per spectrum: about two blocks per SM in all (one part when spectra suffice)
        int dev = 0, sms = 152;
        if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const int S = (int)std::max(1LL, std::min(16LL, 2LL * sms / spectra));
        const unsigned blocks = (unsigned)(spectra * S);
        if (smem > 48 * 1024) {
            cudaError_t e = build == 0 ? cudaFuncSetAttribute(k_build_small<0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                              (int)smem)
                                       : cudaFuncSetAttribute(k_build_small<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                              (int)smem);
            if (e != cudaSuccess) return e;
        }
        if (build == 0)
            k_build_small<0><<<blocks, 256, smem, st>>>(g, ch, S);
        else
            k_build_small<1><<<blocks, 256, smem, st>>>(g, ch, S);
        return cudaGetLastError();
    }
    if (ch.n_tasks == 0) return cudaSuccess;
    if (ch.phi64 || ch.phi32) {
        const long long walks = 2LL * ch.NG * (build == 0 ? g.G : (g.G + 1) / 2);
        const unsigned wblocks = (unsigned)((walks + 3) / 4);
        const int units = build == 0 ? ch.NG : (ch.NG + 1) / 2;  // a warp's cells: one group, or two
        const int warps = std::min(units, 8), gblocks = (units + warps - 1) / warps;
        const unsigned eblocks = (unsigned)((long long)g.n_pieces * gblocks);
        if (build == 0) {
            k_prefix64<<<wblocks, 128, 0, st>>>(g, ch);
            if (eblocks) k_elem64<<<eblocks, warps * 32, 0, st>>>(g, ch, gblocks);
        } else {
            k_prefix32<<<wblocks, 128, 0, st>>>(g, ch);
            if (eblocks) k_elem32<<<eblocks, warps * 32, 0, st>>>(g, ch, gblocks);
        }
        return cudaGetLastError();
    }
    // one warp per task (measured: a persistent launch with a task counter is no faster)
    auto kern = build == 0 ? k_build<0> : (g.pat_prefetch ? k_build<1, true> : k_build<1, false>);
    kern<<<(unsigned)((ch.n_tasks + 3) / 4), 128, 0, st>>>(g, ch);
    return cudaGetLastError();
}

}  // namespace heat
