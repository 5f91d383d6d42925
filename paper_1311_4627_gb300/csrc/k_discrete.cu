// Thermal-discrete cooling (the approximation named beside Eq. adjacent) on the exact path:
// downward rates to every lower bin, and the stationary state of the full rate matrix
// (Eq. steady-state with Eq. level-sum) instead of the Guhathakurta-Draine recursion, which
// needs the adjacent-only cooling of Eq. adjacent.
//
//   k_cooling_window  (grain set-up, once): T_lu = P_emit(T_u; window of l) / (E_u - E_l),
//       the power of Eq. cooling's integrand at T_u in the photon energies that take a grain
//       from bin u to bin l, E in [E_u - Ehi_l, E_u - Elo_l] (l = u-1: [0, E_u - Elo_{u-1}],
//       photons too soft to leave bin u included); the windows tile [0, E_u], so the rates
//       carry the power Eq. cooling's adjacent rate carries.
//   k_td_edges, k_td_env  (once per grain set): where the windows' edges fall on the grid, and
//       which elements of a grain's rate matrix the state reduction touches.
//   k_td_fill  (per spectrum): the rate matrix q[i][j] (from i to j): heating elements
//       T_ji, j > i, as closed-form integrals over the target bin's wavelength window of the
//       log-log interpolant of Omega = u C (plus the intra-bin term on j = i + 1), downward
//       rates from the grain's table; and the absorbed power for the energy check.
//   k_gth  (per spectrum): state reduction (Grassmann, Taksar, Heyman): states n = M..1 are
//       removed, their rates redistributed, q_ij += q_in q_nj / s_n with s_n = sum_{j<n} q_nj
//       (sums and products of non-negative numbers only); then X_0 = 1,
//       X_n = sum_{i<n} X_i q_in / s_n, power-of-two rescales, P = X / sum X.  About M^3/3
//       fused multiply-adds per spectrum, on the FP64 unit, less where rates reach few bins: a
//       block per spectrum, or a cluster of up to eight where a launch has few; states removed
//       in panels of eight (kGthB), q in device memory, read and written once per panel.
#include <algorithm>

#include "common.cuh"
#include "gth_tile.cuh"
#include "internal.h"
#include "rcp64.cuh"
#include "seg64.cuh"

namespace heat {

namespace {

constexpr double kPi = 3.141592653589793;

// Gauss-Legendre (the set-up's nodes, shared with k_cooling) over [ya, yb] in ln(lambda) of
// C(lambda) B_lambda(T) lambda with C = c0 (lambda/lam0)^s.
__device__ double gl_panel(double ya, double yb, double c0, double lam0, double s, double T, const double* glx,
                           const double* glw) {
    double m = 0.5 * (ya + yb), r = 0.5 * (yb - ya), acc = 0.0;
    for (int k = 0; k < kGLPoints; ++k) {
        const double lam = exp(m + r * glx[k]);
        const double x = kHC / (lam * kK * T);
        if (x > 745.0) continue;
        const double l2 = lam * lam;
        const double bl = 2.0 * kH * kC * kC / (l2 * l2 * lam) / expm1(x);
        acc += glw[k] * c0 * pow(lam / lam0, s) * bl * lam;
    }
    return acc * r;
}

// The same over [ya, yb] in sub-panels short enough for the Wien factor: d ln(integrand) /
// d ln(lambda) is about x - 4 + s with x = hc/(lambda k T), so a step of 2/max(x, 4) in
// ln(lambda) keeps each sub-panel within a few e-folds, and every window, however far into the
// tail, is integrated to its own relative accuracy.
__device__ double window_panel(double ya, double yb, double c0, double lam0, double s, double T,
                               const double* glx, const double* glw) {
    double acc = 0.0;
    for (double y = ya; y < yb;) {
        const double x = kHC / (exp(y) * kK * T);
        double h = 2.0 / fmax(x, 4.0);
        if (h > 0.25) h = 0.25;
        const double y1 = y + h < yb ? y + h : yb;
        acc += gl_panel(y, y1, c0, lam0, s, T, glx, glw);
        y = y1;
    }
    return acc;
}

// C(lambda): the log-log interpolant of the nodes, continued beyond the grid with the end
// segments' power laws (as the cooling integral takes it).
__device__ double cabs_at(int N, const double* lam, const double* C, double x) {
    int n;
    if (x < lam[0]) {
        n = 0;
    } else {
        int lo = 0, hi = N - 2;  // last segment with lam[n] <= x
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (lam[mid] <= x) lo = mid; else hi = mid - 1;
        }
        n = lo;
    }
    if (!(C[n] > 0.0 && C[n + 1] > 0.0)) return 0.0;
    return C[n] * pow(x / lam[n], log(C[n + 1] / C[n]) / log(lam[n + 1] / lam[n]));
}

// A narrow window written in the grain's energy after the emission, e in [e0, e0 + de]
// (photon energy E_u - e): its width is exact where it is a tiny fraction of the photon
// energy, which a difference of photon-energy limits would lose.  Gauss-Legendre pieces
// between the grid nodes inside.  Returns int C(E) E^3 / (e^(E/kT) - 1) dE over the window.
__device__ double narrow_window(int N, const double* lam, const double* C, double T, double Eu, double e0, double de,
                                const double* glx, const double* glw) {
    // nodes inside: photon energies hc/lam_n in (Eu - e0 - de, Eu - e0)
    double cuts[6];
    int nc = 0;
    cuts[nc++] = 0.0;
    for (int n = 0; n < N && nc < 5; ++n) {
        const double o = (Eu - kHC / lam[n]) - e0;
        if (o > 0.0 && o < de) cuts[nc++] = o;
    }
    cuts[nc++] = de;
    for (int i = 1; i < nc; ++i) {  // ascending
        const double v = cuts[i];
        int k = i - 1;
        while (k >= 0 && cuts[k] > v) {
            cuts[k + 1] = cuts[k];
            --k;
        }
        cuts[k + 1] = v;
    }
    double acc = 0.0;
    for (int i = 0; i + 1 < nc; ++i) {
        const double r = 0.5 * (cuts[i + 1] - cuts[i]), m = cuts[i] + r;
        if (!(r > 0.0)) continue;
        double s = 0.0;
        for (int k = 0; k < kGLPoints; ++k) {
            const double eps = Eu - (e0 + m + r * glx[k]);
            const double x = eps / (kK * T);
            if (!(eps > 0.0) || x > 745.0) continue;
            s += glw[k] * cabs_at(N, lam, C, kHC / eps) * eps * eps * eps / expm1(x);
        }
        acc += s * r;
    }
    return acc;
}

}  // namespace

// One warp per window (grain g, upper bin u, lower bin l < u); windows of grain g are
// numbered k = u(u-1)/2 + l from woff[g].  Panels as k_cooling's (each grid segment, and
// 0.25 in ln(lambda) beyond the grid with the end segments' power laws), clipped to the
// window's wavelengths [hc/Emax, hc/Emin].
__global__ void k_cooling_window(int N, const double* __restrict__ lam, const double* __restrict__ cabs,
                                 const int* __restrict__ bin_off, int G, const double* __restrict__ T,
                                 const double* __restrict__ E, const long long* __restrict__ woff,
                                 const long long* __restrict__ doff, double* __restrict__ D, const double* glx,
                                 const double* glw) {
    const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= woff[G]) return;
    int g = 0;
    {
        int lo = 0, hi = G - 1;  // last g with woff[g] <= w
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (woff[mid] <= w) lo = mid; else hi = mid - 1;
        }
        g = lo;
    }
    const long long k = w - woff[g];
    int u = (int)floor((1.0 + sqrt(1.0 + 8.0 * (double)k)) * 0.5);
    while ((long long)u * (u - 1) / 2 > k) --u;
    while ((long long)(u + 1) * u / 2 <= k) ++u;
    const int l = (int)(k - (long long)u * (u - 1) / 2);
    const int off = bin_off[g], nb = bin_off[g + 1] - off;
    const double* Eg = E + off;
    const double Tu = T[off + u];
    const double elo_l = l == 0 ? 0.0 : 0.5 * (Eg[l - 1] + Eg[l]);
    const double ehi_l = 0.5 * (Eg[l] + Eg[l + 1]);
    const double emin = l == u - 1 ? 0.0 : Eg[u] - ehi_l;
    const double emax = Eg[u] - elo_l;
    // wavelengths of the window, cut where the integrand is below 1e-340 of its scale
    double lo = kHC / emax;
    const double lmin = kHC / (800.0 * kK * Tu);
    if (lo < lmin) lo = lmin;
    const double hi = emin > 0.0 ? kHC / emin : INFINITY;
    const double* C = cabs + (size_t)g * N;
    if (l < u - 1 && ehi_l - elo_l < 1e-2 * emin) {  // narrow: in the grain's final energy
        if (lane == 0) {
            const double p = 8.0 * kPi / (kH * kH * kH * kC * kC) *
                             narrow_window(N, lam, C, Tu, Eg[u], elo_l, ehi_l - elo_l, glx, glw);
            D[doff[g] + (size_t)u * nb + l] = p / (Eg[u] - Eg[l]);
        }
        return;
    }
    double acc = 0.0;
    if (hi > lo) {
        for (int n = lane; n < N - 1; n += 32) {  // grid segments
            const double a = lam[n], b = lam[n + 1];
            if (b <= lo || a >= hi || !(C[n] > 0.0 && C[n + 1] > 0.0)) continue;
            const double s = log(C[n + 1] / C[n]) / log(b / a);
            acc += window_panel(log(a > lo ? a : lo), log(b < hi ? b : hi), C[n], a, s, Tu, glx, glw);
        }
        if (C[N - 2] > 0.0 && C[N - 1] > 0.0 && hi > lam[N - 1]) {  // past the last node
            const double s = log(C[N - 1] / C[N - 2]) / log(lam[N - 1] / lam[N - 2]);
            const double y0 = log(lam[N - 1] > lo ? lam[N - 1] : lo);
            const double y1 = hi < INFINITY ? log(hi) : y0 + 25.0;
            for (int k2 = lane; y0 + 0.25 * k2 < y1; k2 += 32) {
                const double yb = y0 + 0.25 * (k2 + 1);
                acc += window_panel(y0 + 0.25 * k2, yb < y1 ? yb : y1, C[N - 1], lam[N - 1], s, Tu, glx, glw);
            }
        }
        if (lo < lam[0] && C[0] > 0.0 && C[1] > 0.0) {  // below the first node
            const double s = log(C[1] / C[0]) / log(lam[1] / lam[0]);
            const double ytop = log(hi < lam[0] ? hi : lam[0]), ybot = log(lo);
            for (int k2 = lane; ytop - 0.25 * k2 > ybot; k2 += 32) {
                const double yb = ytop - 0.25 * k2;
                double ya = yb - 0.25;
                if (ya < ybot) ya = ybot;
                acc += window_panel(ya, yb, C[0], lam[0], s, Tu, glx, glw);
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) D[doff[g] + (size_t)u * nb + l] = 4.0 * kPi * acc / (Eg[u] - Eg[l]);
}

// Where the transition wavelength hc / (Elo_f - E_j) of every band element (f, j) falls on the grid: its segment n
// and offset (n = -1 below the grid, N - 1 at or beyond the last node).  Once per grain set; a warp per row f.
__global__ void __launch_bounds__(128) k_td_edges(GrainDev gd, TdEdge* __restrict__ edge) {
    const int w = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (w >= gd.nbt) return;
    int g = 0;
    while (gd.bin_off[g + 1] <= w) ++g;
    const int off = gd.bin_off[g], f = w - off, N = gd.N;
    if (f == 0) return;
    const int e0 = gd.rowptr[off + g + f], wd = gd.rowptr[off + g + f + 1] - e0;
    const double* E = gd.E + off;
    const double elo = 0.5 * (E[f - 1] + E[f]);
    for (int k = lane; k < wd; k += 32) {
        const double x = kHC / (elo - E[f - wd + k]);
        TdEdge r;
        r.n = -1;
        r.t = 0.0;
        r.tau = 0;
        if (x >= gd.lam[N - 1]) {
            r.n = N - 1;
        } else if (x >= gd.lam[0]) {
            int lo = 0, hi = N - 2;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (gd.lam[mid] <= x) lo = mid; else hi = mid - 1;
            }
            r.n = lo;
            r.t = log(x / gd.lam[lo]);
            r.tau = to_q60(fmin(r.t / gd.dln[lo], 1.0));
        }
        edge[e0 + k] = r;
    }
}

cudaError_t launch_td_edges(const GrainDev& g, TdEdge* edge, cudaStream_t st) {
    k_td_edges<<<(unsigned)((g.nbt + 3) / 4), 128, 0, st>>>(g, edge);
    return cudaGetLastError();
}

// Structure of every grain's rate matrix under the state reduction (once per grain set): states are removed from the
// top in panels of kGthB (panel p: states p0 .. hi = nb - 1 - kGthB p), and env[p] holds the lowest row with a
// rate into panel p or a higher one (x), the lowest column its rows reach (y), and the number of panels from
// p on whose rows have only the next lower column (z; 0 for a panel with any other).  Removing a
// panel fills rows [x, p0) with its columns [y, p0), which counts for the panels below.  wmax: the most rows (0) and
// columns (1) below a panel with z = 0; wmax[2 + g]: about how many cycles grain g's reduction takes.  A block per grain.
__global__ void __launch_bounds__(256) k_td_env(GrainDev gd, const double* __restrict__ Dt,
                                                const long long* __restrict__ doff, int4* __restrict__ env,
                                                int* __restrict__ wmax) {
    __shared__ int jl[kDiscreteMaxBins], lo[kDiscreteMaxBins];
    const int g = blockIdx.x, off = gd.bin_off[g], nb = gd.bin_off[g + 1] - off;
    if (nb > kDiscreteMaxBins) return;  // such sets are refused before the solve
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const double* Dg = Dt + doff[g];
    for (int k = 1 + warp; k < nb; k += nw) {
        int j0 = k - 1;
        for (int j = lane; j < k; j += 32)
            if (Dg[(size_t)k * nb + j] != 0.0) {
                j0 = min(j0, j);
                break;
            }
        j0 = __reduce_min_sync(0xffffffffu, j0);
        if (lane == 0) {
            jl[k] = j0;
            lo[k] = min(k - 1, k - (gd.rowptr[off + g + k + 1] - gd.rowptr[off + g + k]));
        }
    }
    __syncthreads();
    if (warp != 0) return;
    int4* ev = env + (off / kGthB + g);
    const int np = (nb - 1 + kGthB - 1) / kGthB;
    int low = nb, rw = 0, cw = 0;
    long long cost = 300LL * nb;
    for (int p = 0; p < np; ++p) {
        const int hi = nb - 1 - kGthB * p, p0 = max(1, hi - kGthB + 1), k = p0 + lane;
        const bool in = k <= hi;
        low = min(low, __reduce_min_sync(0xffffffffu, in ? lo[k] : nb));
        const int jp = __reduce_min_sync(0xffffffffu, in ? jl[k] : nb);
        const bool adj = __all_sync(0xffffffffu, !in || jl[k] == k - 1);
        if (lane == 0) ev[p] = make_int4(low, jp, adj ? 1 : 0, 0);
        if (!adj) {
            rw = max(rw, p0 - low);
            cw = max(cw, p0 - jp);
            cost += 12000 + 4LL * (p0 - low) * (p0 - jp);  // the serial part, kGthB multiply-adds per element
            for (int i = low + lane; i < p0; i += 32)
                if (i > 0) jl[i] = min(jl[i], jp);
        }
        __syncwarp();
    }
    if (lane == 0) {
        for (int p = np - 2; p >= 0; --p)
            if (ev[p].z) ev[p].z = ev[p + 1].z + 1;
        atomicMax(&wmax[0], rw);
        atomicMax(&wmax[1], cw);
        wmax[2 + g] = (int)min(cost, 1LL << 30);
    }
}

cudaError_t launch_td_env(const GrainDev& g, const double* D, const long long* doff, int4* env, int* wmax,
                          cudaStream_t st) {
    k_td_env<<<(unsigned)g.G, 256, 0, st>>>(g, D, doff, env, wmax);
    return cudaGetLastError();
}

// Shared memory of k_td_fill for a grid of N wavelengths, per segment: the cell's A = Omega_n lambda_n^2 dln / h,
// Z = (slope + 2) dln in Q60 (kNoQ60: |Z| >= 1), the segment's integral W = A E1(Z) and the suffix sums of the integrals of
// Omega; and the sums of W over aligned blocks of 8 segments.
size_t td_fill_smem_bytes(int N) { return 32 * (size_t)N + 8 * (((size_t)N + 7) / 8); }
constexpr int64_t kNoQ60 = INT64_MIN;

// Spectrum of block b of a launch that starts at spectrum s0: grains in the order `gorder`
// (longest state reduction first), every cell of the chunk for each grain in turn, so that the spectra of one
// launch have similar cost and the largest start first.
__device__ __forceinline__ void td_spectrum(const ChunkDev& ch, const int* gorder, long long s0, int b, int& cell,
                                            int& g) {
    const long long sp = s0 + b;
    cell = (int)(sp % ch.cells);
    g = gorder[sp / ch.cells];
}

// S blocks per spectrum (cell, grain) of the chunk's cells, each the rows i = part (mod S): q
// [nb][nb] (row-major, rate from row to column) at q + spectrum * qstride, the elements that the state reduction
// touches (env), and the absorbed power c int Omega on the grid (part 0).
// Downward rates are copied from the grain's table (Dt[u][l], from u to l).  The heating
// rate from i into bin j > i is (1/h) int Omega lambda over the photon wavelengths that end in
// bin j, [hc/(Ehi_j - E_i), hc/(Elo_j - E_i)] (Ehi_M = infinity), plus on j = i + 1 the
// power of the photons too soft to leave bin i, c int_{lambda > hc/(Elo_j - E_i)} Omega,
// over E_j - E_i.  The window's edges are the band's transition wavelengths (j + 1, i) and (j, i), whose places on
// the grid do not depend on the cell (edge table).  A row's windows tile the grid: each is its
// partial end segments plus the segment integrals between them (summed, by eights, not differenced; inside one segment
// a difference of two Q60 values, to 2^-53 of the segment); the soft term is its partial segment plus
// a suffix sum.  A warp per row, a lane per j; neighbouring lanes share their window edge, so a window costs one
// fixed-point E1 (seg64.cuh).  With the edges and each partial segment's logarithms and exponentials in FP64
// the fill was bound by the FP64 unit (83 % busy): 8 cells x 64 grains x 1024 wavelengths 8.7 ms, then
// 2.0 ms, bound by the lanes whose window spans a hundred segments; with the sums by eights 0.64 ms.
__global__ void __launch_bounds__(256) k_td_fill(GrainDev gd, ChunkDev ch, const double* __restrict__ Dt,
                                                 const long long* __restrict__ doff, const int* __restrict__ gorder,
                                                 const TdEdge* __restrict__ edge, const int4* __restrict__ env,
                                                 long long s0, double* q, long long qstride, int S) {
    extern __shared__ double fsm[];
    const int bsp = blockIdx.x / S, part = blockIdx.x % S;  // spectrum of the launch, part of its rows
    int cell, g;
    td_spectrum(ch, gorder, s0, bsp, cell, g);
    const int N = gd.N;
    double* A = fsm;
    int64_t* Z = (int64_t*)(A + N);
    double* W = (double*)(Z + N);
    double* S0 = W + N;
    double* W8 = S0 + N;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    for (int n = tid; n < N; n += blockDim.x) {
        double a = 0.0, i0 = 0.0, w = 0.0;
        int64_t z = 0;
        if (n < N - 1) {
            const size_t gn = (size_t)g * N + n;
            const double ua = ch.ua64[(size_t)n * ch.Cc + cell], su = ch.su64[(size_t)n * ch.Cc + cell];
            const double dl = gd.dln[n], q1 = su + gd.sC[gn] + 2.0, zd = q1 * dl;
            a = ua * gd.ca64[gn] * dl;
            if (a > 0.0) {
                i0 = add_segment(0.0, ua * gd.ce64[gn], q1 - 1.0, dl);
                const int cls = e1_class(zd);
                if (cls) {
                    z = to_q60(zd);
                    w = a * from_q60(e1_q60(cls, z));
                } else {
                    z = kNoQ60;
                    w = a * e1d(zd);
                }
            } else {
                a = 0.0;
            }
        }
        A[n] = a;
        Z[n] = z;
        W[n] = w;
        S0[n] = i0;
    }
    __syncthreads();
    for (int b = tid; b < (N + 7) / 8; b += blockDim.x) {
        double w = 0.0;
        for (int n = 8 * b; n < min(N, 8 * b + 8); ++n) w += W[n];
        W8[b] = w;
    }
    if (warp == 0) {  // suffix sums of the segment integrals of Omega, S0[n] = sum_{m >= n}
        const int per = (N + 31) / 32, b0 = lane * per, b1 = min(N, b0 + per);
        double part = 0.0;
        for (int n = b1 - 1; n >= b0; --n) part += S0[n];
        double above = 0.0;  // sum over the lanes after this one
        for (int o = 1; o < 32; o <<= 1) {
            const double t = __shfl_down_sync(0xffffffffu, part + above, o);
            if (lane + o < 32) above += t;
        }
        for (int n = b1 - 1; n >= b0; --n) {
            above += S0[n];
            S0[n] = above;
        }
    }
    __syncthreads();
    const int off = gd.bin_off[g], nb = gd.bin_off[g + 1] - off;
    const double* Dg = Dt + doff[g];
    const int* rp = gd.rowptr + off + g;
    const int4* ev = env + (off / kGthB + g);
    const int np = (nb - 1 + kGthB - 1) / kGthB;
    double* qs = q + (size_t)bsp * qstride;
    // the cell's slope + 2 of segment n (only where |Z| >= 1)
    auto slope = [&](int n) { return ch.su64[(size_t)n * ch.Cc + cell] + gd.sC[(size_t)g * N + n] + 2.0; };
    // tau E1(Z tau) in Q60: the fraction of A up to an edge in segment n
    auto upto = [&](int n, int64_t tau) -> int64_t {
        const int64_t z = Z[n];
        if (z == kNoQ60) return 0;
        const int64_t az = z < 0 ? -z : z;
        return mul_q60(tau, e1_q60(az < (kQ60 >> 4) ? 3 : az < (kQ60 >> 2) ? 2 : 1, mul_q60(z, tau)));
    };
    // sum of the whole segments n0 .. n1 - 1
    auto wholes = [&](int n0, int n1) {
        double v = 0.0;
        int n = n0;
        for (; n < n1 && (n & 7); ++n) v += W[n];
#pragma unroll 4
        for (; n + 8 <= n1; n += 8) v += W8[n >> 3];
        for (; n < n1; ++n) v += W[n];
        return v;
    };
    // integral between offsets ta and tb of segment n (r: upto() of both)
    auto between = [&](int n, double ta, double tb, int64_t ra, int64_t rb) {
        if (A[n] == 0.0) return 0.0;
        if (Z[n] != kNoQ60) return rb > ra ? A[n] * from_q60(rb - ra) : 0.0;
        const double q1 = slope(n);
        return A[n] / (q1 * gd.dln[n]) * exp(q1 * ta) * expm1(q1 * (tb - ta));
    };
    for (int i = part + S * warp; i < nb; i += S * nw) {
        double* qi = qs + (size_t)i * nb;
        const double* di = Dg + (size_t)i * nb;
        const int p = min((nb - 1 - i) / kGthB, np - 1);  // row 0 is in no panel: its first column is its own
        for (int j = (i == 0 ? 0 : ev[p].z ? i - 1 : ev[p].y) + lane; j <= i; j += 32) qi[j] = j < i ? di[j] : 0.0;
        int reach = i;  // the row's last column
        for (int pb = 0; pb < np; pb += 32) {
            const unsigned m = __ballot_sync(0xffffffffu, pb + lane < np && ev[min(pb + lane, np - 1)].x <= i);
            if (m) {
                reach = nb - 1 - kGthB * (pb + __ffs(m) - 1);
                break;
            }
        }
        for (int jb = i + 1; jb <= reach; jb += 32) {
            const int j = jb + lane;
            // the window's long-wavelength edge, element (j, i); n = -1: below the grid (or no such bin)
            auto edge_of = [&](int jj) {
                TdEdge r;
                r.n = -1;
                r.t = 0.0;
                r.tau = 0;
                if (jj < nb) {
                    const int p0 = rp[jj], p1 = rp[jj + 1];
                    const int k = i - (jj - (p1 - p0));
                    if (k >= 0) r = edge[p0 + k];
                }
                return r;
            };
            const TdEdge b = edge_of(j);
            const int64_t rb = b.n >= 0 && b.n < N - 1 ? upto(b.n, b.tau) : 0;
            // the other edge is the next lane's
            TdEdge a;
            a.n = __shfl_down_sync(0xffffffffu, b.n, 1);
            a.t = __shfl_down_sync(0xffffffffu, b.t, 1);
            int64_t ra = __shfl_down_sync(0xffffffffu, (long long)rb, 1);
            if (lane == 31) {
                a = edge_of(j + 1);
                ra = a.n >= 0 && a.n < N - 1 ? upto(a.n, a.tau) : 0;
            }
            if (a.n < 0) {  // from the grid's short end
                a.n = 0;
                a.t = 0.0;
                ra = 0;
            }
            if (j <= reach) {
                double v = 0.0;
                if (b.n >= 0) {
                    if (a.n == b.n) {
                        if (b.n < N - 1) v = between(b.n, a.t, b.t, ra, rb);
                    } else {
                        v = between(a.n, a.t, gd.dln[a.n], ra, upto(a.n, kQ60)) + wholes(a.n + 1, b.n);
                        if (b.n < N - 1) v += between(b.n, 0.0, b.t, 0, rb);
                    }
                }
                if (j == i + 1 && b.n < N - 1) {  // photons too soft to leave bin i
                    const double ide = gd.invdE[off + i];
                    v += b.n < 0 ? soft_end(S0[0], ide)
                                 : soft_term(gd, g, b.n, ch.ua64[(size_t)b.n * ch.Cc + cell],
                                             ch.su64[(size_t)b.n * ch.Cc + cell], b.t, b.tau, S0[b.n + 1], ide);
                }
                qi[j] = v;
            }
        }
    }
    if (tid == 0 && part == 0 && ch.pabs) ch.pabs[(size_t)cell * gd.G + g] = kC * S0[0];
}

namespace {

__device__ __forceinline__ double block_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < 32) {
        t = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) red[0] = t;
    }
    __syncthreads();
    return red[0];
}

}  // namespace

namespace {

// 1/s as kept for the back substitution: -1 where nothing leaves a state downward.  Comparisons are on the bits:
// the FP64 unit takes 64 cycles for one too.
__device__ __forceinline__ double exit_of(double s, double r) { return __double_as_longlong(s) == 0 ? -1.0 : r; }

template <bool CLUSTER>
__device__ __forceinline__ void gth_sync() {
    if (CLUSTER)
        asm volatile(
            "barrier.cluster.arrive.release;\n\t"
            "barrier.cluster.wait.acquire;" ::
                : "memory");
    else
        __syncthreads();
}

}  // namespace

// Shared memory of k_gth: 1/s and X [nb], the panel's rows below it [kGthB][cw], the rows' panel columns
// [rcap][kGthB], the panel table.
size_t gth_smem_bytes(int max_bins, int rcap, int cw) {
    const int np = (max_bins + kGthB - 1) / kGthB;
    return sizeof(double) * (2 * (size_t)max_bins + (size_t)kGthB * cw + (size_t)kGthB * rcap + 2) +
           sizeof(int4) * (size_t)np;
}

// One block (CLUSTER: a cluster of C blocks) per spectrum: state reduction of q, back substitution, P and the
// energy check.
//
// States are removed from the top; removing state k, with s_k = sum_{j < k} q_kj, adds q_ik q_kj / s_k to q_ij
// for i, j < k.  Every term is a product of non-negative numbers.  kGthB states [p0, hi] are removed at a time:
//  - The panel by itself: its kGthB x kGthB block and, per row, the sums R(m) of the elements below column m
//    (the row's sum below the panel and the block's lower part).  They are updated like
//    elements, R_i(m) += (q_ik / s_k) R_k(m) for m <= i, so s_k = R_k(k) is at hand when k's turn comes without a sum
//    over the row and without the rest of the row.  One warp, four numbers a lane, no barrier: per state the
//    chain is a shuffle, a reciprocal, a multiply and a multiply-add (about 500 cycles).
//  - Then, with the panel's multipliers known, its rows below the panel, a thread per column, and the
//    panel's columns of the rows below, a thread per row.
//  - Then the block below: q_ij += sum_k (q_ik / s_k) q_kj, a warp per two rows and 32 columns.
// Rows that do not reach the panel and columns it does not reach are left out (env).  A run of panels whose rows
// have only the next lower column (grains whose levels are wider than the photons they emit) fills nothing below the
// diagonal: all its s_k = q_k,k-1 are known at once, and removing k moves q_ik to q_i,k-1, a thread per row.
//
// Back substitution: X_0 = 1, X_n = sum_{i < n} X_i q_in / s_n, in ascending i, 32 states at a time: one warp
// through the 32 x 32 block in shared memory (a lane per column; multiply, shuffle, multiply-add per state), then all
// threads add the 32 rows to the columns beyond.  Past 2^800 every X is scaled by 2^-800 (exact).  P = X / sum X.
//
// Removing state by state with a barrier, a sum over the row and a division each took 5,000 cycles a state at
// 128 bins, two thirds of them waiting: 8 spectra x 128 bins 431 us, now 186 us; 512 spectra of 128 ..
// 1024 bins 7.7 ms, now 1.2 ms.  At 128 bins, where every rate is non-zero, one block is bound by its
// SM's FP64 unit (183 us for the nb^3 / 3 multiply-adds), hence the cluster when a launch has few spectra:
// rows below a panel go round the blocks in pairs, and each block repeats the panel's own part.
template <bool CLUSTER>
__global__ void __launch_bounds__(kGthThreads, 2) k_gth(GrainDev gd, ChunkDev ch, const int* __restrict__ gorder,
                                                        const int4* __restrict__ env, int rcap, int cw, int C,
                                                        long long s0, double* q, long long qstride) {
    extern __shared__ __align__(16) double smd[];
    __shared__ double red[kGthThreads / 32];
    __shared__ double tile[32][32];
    __shared__ double As[kGthB][kGthB], CL[kGthB][kGthB], UA[kGthB][kGthB], Rs[kGthB], rk[kGthB];
    constexpr int nw = kGthThreads / 32;
    static_assert(kGthB == 8 && nw >= kGthB, "k_gth: a warp per panel row, four numbers of the panel per lane");
    const int rank = CLUSTER ? (int)(blockIdx.x % C) : 0, sp = CLUSTER ? (int)(blockIdx.x / C) : (int)blockIdx.x;
    const int nC = CLUSTER ? C : 1;
    int cell, g;
    td_spectrum(ch, gorder, s0, sp, cell, g);
    const int off = gd.bin_off[g], nb = gd.bin_off[g + 1] - off;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double* Ls = smd;                      // [rcap][kGthB], rcap even
    double* U = Ls + (size_t)rcap * kGthB;  // [kGthB][cw]
    double* rs = U + (size_t)kGthB * cw;
    double* X = rs + nb;
    int4* ev = (int4*)(X + nb);  // an even number of doubles before it
    double* qs = q + (size_t)sp * qstride;
    const int np = (nb - 1 + kGthB - 1) / kGthB;
    for (int p = tid; p < np; p += kGthThreads) ev[p] = env[off / kGthB + g + p];
    __syncthreads();
    const int pi = lane & 7, pc = lane >> 3;  // the panel in warp 0: row, first column (and + 4)
    double b0 = 0.0, b1 = 0.0;                // the last panel's block above the diagonal, stored one panel late:
    int bp = -1, bn = 0;                              // other blocks of the cluster may still be reading it
    auto store_block = [&]() {
        if (warp == 0 && rank == 0 && bp > 0) {
            double* qr = qs + (size_t)(bp + pi) * nb + bp;
            if (pc > pi && pc < bn) qr[pc] = b0;
            if (pc + 4 > pi && pc + 4 < bn) qr[pc + 4] = b1;
        }
    };
    for (int p = 0; p < np;) {
        const int4 e = ev[p];
        const int hi = nb - 1 - kGthB * p;
        if (e.z > 0) {  // a run of panels with adjacent downward rates only
            const int pe = p + e.z, a = max(1, nb - kGthB * pe), lo = ev[pe - 1].x;
            for (int k = a + tid; k <= hi; k += kGthThreads) {
                const double s = qs[(size_t)k * nb + k - 1];
                rs[k] = exit_of(s, rcp_or_0(s));
            }
            __syncthreads();
            for (int i = lo + rank * kGthThreads + tid; i < hi - 1; i += nC * kGthThreads) {
                int t0 = p, t1 = pe;  // first panel of the run that row i reaches (x falls with the panel)
                while (t0 < t1) {
                    const int m = (t0 + t1) >> 1;
                    if (ev[m].x > i) t0 = m + 1; else t1 = m;
                }
                const int top = nb - 1 - kGthB * t0;
                double* qi = qs + (size_t)i * nb;
                const int bot = max(a, i + 2);
                if (top < bot) continue;
                double x = qi[top];
                for (int k = top; k >= bot; k -= 8) {
                    double v[8];
#pragma unroll
                    for (int t = 0; t < 8; ++t) v[t] = k - t >= bot ? qi[k - t - 1] : 0.0;
#pragma unroll
                    for (int t = 0; t < 8; ++t)
                        if (k - t >= bot) {
                            x = __double2hiint(rs[k - t]) > 0 ? v[t] + x : v[t];
                            qi[k - t - 1] = x;
                        }
                }
            }
            gth_sync<CLUSTER>();
            store_block();
            bp = -1;
            p = pe;
            continue;
        }
        const int p0 = max(1, hi - kGthB + 1), nk = hi - p0 + 1, ilo = e.x, jp = e.y, nc = p0 - jp, nr = p0 - ilo;
        // the panel's block and its rows' sums below it
        if (tid < kGthB * kGthB) {
            const int i = tid >> 3, c = tid & 7;
            As[i][c] = i < nk && c < nk && i != c ? qs[(size_t)(p0 + i) * nb + p0 + c] : 0.0;
        }
        if (warp < kGthB) {
            double s[4] = {0.0, 0.0, 0.0, 0.0};
            if (warp < nk) {
                const double* qk = qs + (size_t)(p0 + warp) * nb;
                for (int j = jp + lane; j < p0; j += 128)
#pragma unroll
                    for (int t = 0; t < 4; ++t) s[t] += j + 32 * t < p0 ? qk[j + 32 * t] : 0.0;
            }
            double t = (s[0] + s[1]) + (s[2] + s[3]);
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane == 0) Rs[warp] = t;
        }
        __syncthreads();
        store_block();
        bp = -1;
        if (warp == 0) {
            double e0 = As[pi][pc], e1 = As[pi][pc + 4], R0 = Rs[pi], R1;
#pragma unroll
            for (int m = 0; m < 3; ++m) R0 = m < pc ? R0 + As[pi][m] : R0;
            R1 = R0;
#pragma unroll
            for (int m = 0; m < 7; ++m) R1 = m >= pc && m < pc + 4 ? R1 + As[pi][m] : R1;
            double rown = 0.0;  // 1/s of this lane's row
#pragma unroll
            for (int k = kGthB - 1; k >= 0; --k) {
                const double s = __shfl_sync(0xffffffffu, k < 4 ? R0 : R1, k | ((k & 3) << 3));
                const double r = rcp_or_0(s);
                if (pi == k) rown = r;
                if (lane == 0 && k < nk) rs[p0 + k] = exit_of(s, r);
                if (k == 0) break;
                const double qik = __shfl_sync(0xffffffffu, k < 4 ? e0 : e1, pi | ((k & 3) << 3));
                const int src = k | (pc << 3);
                const double v0 = __shfl_sync(0xffffffffu, e0, src), u0 = __shfl_sync(0xffffffffu, R0, src);
                const double c = qik * r;
                if (pi < k) {
                    if (pc == 0) CL[pi][k] = c;
                    R0 = fma(c, u0, R0);
                    if (pc < k) e0 = fma(c, v0, e0);
                }
                if (k > 4) {
                    const double v1 = __shfl_sync(0xffffffffu, e1, src), u1 = __shfl_sync(0xffffffffu, R1, src);
                    if (pi < k) {
                        R1 = fma(c, u1, R1);
                        if (pc + 4 < k) e1 = fma(c, v1, e1);
                    }
                }
            }
            UA[pi][pc] = e0 * rown;
            UA[pi][pc + 4] = e1 * rown;
            if (pc == 0) rk[pi] = rown;
            b0 = e0;
            b1 = e1;
            bp = p0;
            bn = nk;
        }
        __syncthreads();
        // rows below the panel: this block's, in pairs
        const int lp_all = (nr + 1) / 2, lp_own = (lp_all - rank + nC - 1) / nC;
        const int ncp = (nc + 31) & ~31;
        for (int l0 = 0; l0 == 0 || l0 < 2 * lp_own; l0 += rcap) {
            const int ln = min(rcap, 2 * lp_own - l0);  // rows of this turn
            auto row_of = [&](int l) { return ilo + 2 * (((l0 + l) >> 1) * nC + rank) + (l & 1); };
            for (int t = (l0 == 0 ? 0 : ncp) + tid; t < ncp + ln; t += kGthThreads) {
                asm volatile("" ::: "memory");  // read the multipliers per turn: they'd fill the registers
                if (t < ncp) {  // a column of the panel's rows
                    if (t >= nc) continue;
                    double v[kGthB];
#pragma unroll
                    for (int k = 0; k < kGthB; ++k) v[k] = k < nk ? qs[(size_t)(p0 + k) * nb + jp + t] : 0.0;
#pragma unroll
                    for (int k = kGthB - 1; k > 0; --k)
#pragma unroll
                        for (int i = 0; i < k; ++i) v[i] = fma(CL[i][k], v[k], v[i]);
#pragma unroll
                    for (int k = 0; k < kGthB; ++k) U[k * cw + t] = v[k];
                } else {  // a row's panel columns
                    const int l = t - ncp, i = row_of(l);
                    double x[kGthB];
                    double* qi = qs + (size_t)i * nb + p0;
#pragma unroll
                    for (int k = 0; k < kGthB; ++k) x[k] = i < p0 && k < nk ? qi[k] : 0.0;
#pragma unroll
                    for (int k = kGthB - 1; k > 0; --k)
#pragma unroll
                        for (int j = 0; j < k; ++j) x[j] = fma(x[k], UA[k][j], x[j]);
#pragma unroll
                    for (int k = 0; k < kGthB; ++k) {
                        if (i < p0 && k < nk) qi[k] = x[k];
                        Ls[l * kGthB + k] = x[k] * rk[k];
                    }
                }
            }
            __syncthreads();
            // the block below: two rows and 32 columns per warp
            const int ncc = ncp >> 5, nt = ln > 0 ? (ln / 2) * ncc : 0;
            double v0 = 0.0, v1 = 0.0, n0 = 0.0, n1 = 0.0;
            auto load = [&](int t, double& x0, double& x1) {
                const int l = 2 * (t / ncc), j = jp + 32 * (t % ncc) + lane, i = row_of(l);
                if (t < nt && j < p0) {
                    x0 = qs[(size_t)i * nb + j];
                    if (i + 1 < p0) x1 = qs[(size_t)(i + 1) * nb + j];
                }
            };
            if (nt > 0) load(warp, n0, n1);
            for (int t = warp; t < nt; t += nw) {
                v0 = n0;
                v1 = n1;
                load(t + nw, n0, n1);
                const int l = 2 * (t / ncc), cj = 32 * (t % ncc) + lane, i = row_of(l);
                const double2* L0 = (const double2*)(Ls + l * kGthB);
                const double* Uj = U + min(cj, nc - 1);
#pragma unroll
                for (int k = kGthB - 2; k >= 0; k -= 2) {
                    const double2 a = L0[k >> 1], b = L0[(k >> 1) + kGthB / 2];
                    const double uh = Uj[(k + 1) * cw], ul = Uj[k * cw];
                    v0 = fma(a.y, uh, v0);
                    v1 = fma(b.y, uh, v1);
                    v0 = fma(a.x, ul, v0);
                    v1 = fma(b.x, ul, v1);
                }
                if (cj < nc) {
                    qs[(size_t)i * nb + jp + cj] = v0;
                    if (i + 1 < p0) qs[(size_t)(i + 1) * nb + jp + cj] = v1;
                }
            }
            if (l0 + rcap < 2 * lp_own) __syncthreads();
        }
        gth_sync<CLUSTER>();
        ++p;
    }
    store_block();
    if (rank != 0) return;
    // back substitution (X holds the sums so far beyond the current block)
    for (int n = tid; n < nb; n += kGthThreads) X[n] = n == 0 ? 1.0 : 0.0;
    if (tid == 0) rs[0] = 1.0;
    __syncthreads();
    bool bad = false;
    auto low_of = [&](int n) { return n == 0 ? 0 : ev[(nb - 1 - n) / kGthB].x; };
    for (int n0 = 0; n0 < nb; n0 += 32) {
        const int n = n0 + lane;
        const bool in = n < nb;
        const int low = in ? low_of(n) : nb;
#pragma unroll
        for (int i = warp; i < 32; i += nw)
            tile[i][lane] = gth_tile_in(i, lane, n0, nb, low) ? qs[(size_t)(n0 + i) * nb + n] : 0.0;
        __syncthreads();
        if (warp == 0) {
            double x = in ? X[n] : 0.0;
            const double r = in ? rs[n] : 0.0;
#pragma unroll 8
            for (int i = 0; i < 32; ++i) {
                double xi = x * r;  // lane i: every state below it has contributed
                if (lane == i) {
                    if (__double2hiint(r) < 0) {
                        bad |= x != 0.0;
                        xi = 0.0;
                    }
                    x = xi;
                }
                xi = __shfl_sync(0xffffffffu, xi, i);
                if (__double2hiint(xi) >= (1023 + 800) << 20) {
                    xi *= 0x1p-800;
                    x *= 0x1p-800;
                    for (int m = lane; m < nb; m += 32)
                        if (m < n0 || m >= n0 + 32) X[m] *= 0x1p-800;
                }
                if (lane > i) x = fma(xi, tile[i][lane], x);
            }
            if (in) X[n] = x;
        }
        __syncthreads();
        for (int n = n0 + 32 + tid; n < nb; n += kGthThreads) {
            const int low = max(low_of(n), n0);
            if (low >= n0 + 32) break;  // nor do the columns beyond reach down here
            double x = X[n];
#pragma unroll 8
            for (int i = low; i < n0 + 32; ++i) x = fma(X[i], qs[(size_t)i * nb + n], x);
            X[n] = x;
        }
        __syncthreads();
    }
    bad = __syncthreads_or(bad);
    double part = 0.0;
    for (int i = tid; i < nb; i += kGthThreads) part += X[i];
    const double inv = 1.0 / block_sum(part, red);
    double emit = 0.0;
    double* prow = ch.P + (size_t)cell * ch.ldP + off;
    for (int i = tid; i < nb; i += kGthThreads) {
        const double pr = X[i] * inv;
        prow[i] = pr;
        emit = fma(pr, gd.cde[off + i], emit);
    }
    emit = block_sum(emit, red);
    if (tid == 0) {
        if (ch.ledger) {
            double* lg = ch.ledger + ((size_t)cell * gd.G + g) * 2;
            lg[0] = ch.pabs[(size_t)cell * gd.G + g];
            lg[1] = emit;
        }
        if (bad) atomicOr(ch.status, kStatNumeric);
    }
}

cudaError_t launch_cooling_window(int N, const double* lam, const double* cabs, const int* bin_off, int G,
                                  const double* T, const double* E, const long long* woff, long long n_windows,
                                  const long long* doff, double* D, const double* glx, const double* glw,
                                  cudaStream_t st) {
    if (n_windows <= 0) return cudaSuccess;
    const long long threads = n_windows * 32;
    k_cooling_window<<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(N, lam, cabs, bin_off, G, T, E, woff, doff,
                                                                        D, glx, glw);
    return cudaGetLastError();
}

long long discrete_batch_spectra(const GrainDev& g, const ChunkDev& ch, long long s0, long long batch) {
    const long long spectra = (long long)ch.cells * g.G;
    return spectra - s0 < batch ? spectra - s0 : batch;
}

cudaError_t launch_discrete_fill(const GrainDev& g, const ChunkDev& ch, const double* D, const long long* doff,
                                 const int* gorder, const TdEdge* edge, const int4* env, double* q, long long qstride,
                                 long long s0, long long n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const size_t smem = td_fill_smem_bytes(g.N);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_td_fill, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    // parts per spectrum (rows by residue): about two blocks per SM when the launch has few spectra
    int dev = 0, sms = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int S = (int)(n >= 2LL * sms ? 1 : std::min(16LL, std::max(1LL, 2LL * sms / n)));
    k_td_fill<<<(unsigned)(n * S), 256, smem, st>>>(g, ch, D, doff, gorder, edge, env, s0, q, qstride, S);
    return cudaGetLastError();
}

cudaError_t launch_discrete_gth(const GrainDev& g, const ChunkDev& ch, const int* gorder, const int4* env, int rw,
                                int cw, double* q, long long qstride, long long s0, long long n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    int dev = 0, sms = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // Blocks per spectrum: the most that still run at once, where panels have enough rows to share (each block
    // repeats a panel's serial part, so narrow ones gain nothing).
    int C = 1;
    if (rw >= 32)
        while (C < 8 && n * C * 2 <= sms) C *= 2;
    const int rcap = std::min(kGthRows, (rw + 2 * C - 1) / (2 * C) * 2);
    const size_t smem = gth_smem_bytes(g.max_bins, rcap, cw);
    const void* fn = C > 1 ? (const void*)k_gth<true> : (const void*)k_gth<false>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3((unsigned)(n * C));
    lc.blockDim = dim3(kGthThreads);
    lc.dynamicSmemBytes = smem;
    lc.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)C;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    lc.attrs = &at;
    lc.numAttrs = C > 1 ? 1 : 0;
    return C > 1 ? cudaLaunchKernelEx(&lc, k_gth<true>, g, ch, gorder, env, rcap, cw, C, s0, q, qstride)
                 : cudaLaunchKernelEx(&lc, k_gth<false>, g, ch, gorder, env, rcap, cw, C, s0, q, qstride);
}

}  // namespace heat
