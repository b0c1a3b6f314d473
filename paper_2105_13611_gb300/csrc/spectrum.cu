// synth_spectrum: emergent intensity of one model atmosphere (paper Eq. Ilambda,
// LTE source S = B_lambda(T), no scattering).
//
// Per depth the populations (FP64, same kernel as set_atmosphere_grid), the line
// opacity on the window grid (synth_rows, the synth_opacity pipeline) and the
// flat continuum are computed; k_formal then integrates, per wavelength point,
//   tau_0 = kappa_0 m_0, tau_{d+1} = tau_d + (kappa_d + kappa_{d+1})(m_{d+1} - m_d)/2,
//   I_{D-1} = S_{D-1} + mu dS/dtau (diffusion),
//   I_d = I_{d+1} e^{-x} + S_d (1 - e^{-x}) + (S_{d+1} - S_d)(1 - e^{-x}(1 + x))/x,  x = dtau/mu,
//   I = I_0 e^{-tau_0/mu} + S_0 (1 - e^{-tau_0/mu}) at the surface.
//
// odf_intensity: bin intensities of many 1D atmospheres from an ODF table (paper
// Sect. 2.3 and App. E), I_bin = sum_s w_s I_lambda_c(kappa_c + kappa_s): per depth the
// sub-bin opacities and the continuum are interpolated bilinearly in (log10 T, log10 P)
// on the table grid, and each sub-bin's intensity follows from the same formal solution.
#include <math.h>

#include <algorithm>
#include <vector>

#include "common.cuh"
#include "internal.cuh"
#include "voigt.cuh"   // packed FP32

namespace mpsa {

namespace {

constexpr int kMaxDepth = 256;
constexpr int kMaxMu = 16;

// B_lambda(T) = c1 / (e^x - 1), x = c2 / T.  Beyond x = 80 (e^x near the FP32 range) it is
// formed in log space, exp(ln c1 - x), whose dropped term ln(1 - e^-x) is below 2e-35; the
// value then stays representable down to FP32's smallest normal number instead of
// flushing to zero where e^x overflows.
__device__ __forceinline__ float planck_f32(float c1, float lnc1, float c2, float T) {
    const float x = c2 / T;
    return x < 80.f ? c1 / expm1f(x) : expf(lnc1 - x);
}

// 2^y and 1/y by the special-function unit (PTX ex2.approx / rcp.approx; relative error
// near 2^-22)
__device__ __forceinline__ float ex2_fast(float y) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y));
    return r;
}
__device__ __forceinline__ float rcp_fast(float y) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y));
    return r;
}

// e^{-x} and the layer weights ome = 1 - e^{-x}, wl = (1 - e^{-x}(1 + x)) / x of an optical
// thickness x = dtau / mu (rx = 1/x), the last two by their Taylor series below x = 0.1 (no
// cancellation; there a warp's layers are all thin)
__device__ __forceinline__ void layer_weights(float x, float e, float rx, float* ome, float* wl) {
    if (x < 0.1f) {
        // 1 - e^{-x} = x - x^2/2 + x^3/6 - x^4/24 + x^5/120
        *ome = x * fmaf(x, fmaf(x, fmaf(x, fmaf(x, 1.f / 120.f, -1.f / 24.f), 1.f / 6.f), -0.5f), 1.f);
        // (1 - e^{-x}(1 + x))/x = x/2 - x^2/3 + x^3/8 - x^4/30 + x^5/144
        *wl = x * fmaf(x, fmaf(x, fmaf(x, fmaf(x, 1.f / 144.f, -1.f / 30.f), 0.125f), -1.f / 3.f), 0.5f);
    } else {
        *ome = 1.f - e;
        *wl = (1.f - fmaf(e, x, e)) * rx;
    }
}

// k_formal: the emergent intensity of NMU directions at one wavelength point per thread (blockIdx.y
// counts groups of NMU directions).  The recurrence runs from the bottom up and needs only
// the layers' optical thicknesses, so nothing is kept per depth: with tau and S of every
// depth in local memory, and three exponentials per layer and direction, 80 depths x 7300 points x 5
// directions took 134 us, now 54 us.  All directions of a point share its Planck function
// (NMU = 5); a window too narrow to fill the GPU spreads them over threads (NMU = 1; formal_launch).
template <int NMU>
__global__ void __launch_bounds__(128) k_formal(int D, int N, const float* __restrict__ kappa,
                                                const float* __restrict__ kc, const float* __restrict__ kcont,
                                                const float* __restrict__ m, const float* __restrict__ T, double lam0_nm,
                                                double lnq, int n_mu, const float* __restrict__ mu,
                                                float* __restrict__ I_out) {
    __shared__ float sm[kMaxDepth], sT[kMaxDepth], skc[kMaxDepth];
    for (int d = threadIdx.x; d < D; d += blockDim.x) {
        sm[d] = m[d];
        sT[d] = T[d];
        skc[d] = kcont ? 0.f : kc[d];
    }
    __syncthreads();
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    const double lam_cm = lam0_nm * exp((double)j * lnq) * 1e-7;
    const double c1d = 2.0 * kH * kC * kC / (lam_cm * lam_cm * lam_cm * lam_cm * lam_cm);
    const float c1 = (float)c1d, lnc1 = (float)log(c1d);
    const float c2 = (float)(kH * kC / (lam_cm * kKB));
    const int q0 = blockIdx.y * NMU;
    float I[NMU], u[NMU], ru[NMU];
#pragma unroll
    for (int q = 0; q < NMU; ++q) {
        u[q] = q0 + q < n_mu ? mu[q0 + q] : 1.f;
        ru[q] = 1.f / u[q];
    }
    auto total = [&](int d) {   // line opacity and the depth's flat or closed-form continuum
        return kappa[(size_t)d * N + j] + (kcont ? kcont[(size_t)d * N + j] : skc[d]);
    };
    float k_hi = total(D - 1), k_lo = total(D - 2);
    float S_hi = planck_f32(c1, lnc1, c2, sT[D - 1]), S_lo = planck_f32(c1, lnc1, c2, sT[D - 2]);
    float dtau = 0.5f * (k_lo + k_hi) * (sm[D - 1] - sm[D - 2]);
    const float dS = (S_hi - S_lo) / dtau;
#pragma unroll
    for (int q = 0; q < NMU; ++q) I[q] = fmaf(u[q], dS, S_hi);
    for (int d = D - 2;; --d) {
        const float dSl = S_hi - S_lo, rdt = rcp_fast(dtau);
        const float k_next = d > 0 ? total(d - 1) : 0.f;   // in flight while this layer is worked on
#pragma unroll
        for (int q = 0; q < NMU; ++q) {
            const float x = dtau * ru[q];
            const float e = expf(-x);
            float ome, wl;
            layer_weights(x, e, u[q] * rdt, &ome, &wl);
            I[q] = fmaf(I[q], e, fmaf(S_lo, ome, dSl * wl));
        }
        if (d == 0) break;
        k_hi = k_lo;
        k_lo = k_next;
        S_hi = S_lo;
        S_lo = planck_f32(c1, lnc1, c2, sT[d - 1]);
        dtau = 0.5f * (k_lo + k_hi) * (sm[d] - sm[d - 1]);
    }
    const float tau0 = k_lo * sm[0];
#pragma unroll
    for (int q = 0; q < NMU; ++q) {
        const float x0 = tau0 * ru[q];
        if (q0 + q < n_mu) I_out[(size_t)(q0 + q) * N + j] = I[q] * expf(-x0) + S_lo * (-expm1f(-x0));
    }
}

// ---- bin intensities from an ODF table
//
// Three kernels per call:
//  * k_bin_table: the FP64 table rounded once to FP32 (the interpolation then runs on the
//    FP32 pipes; per-value conversions in the main loop kept the FP64 pipe 86 % busy) and
//    turned to [row][sub-bin][bin], the bins padded to an even number;
//  * k_bin_cells: per (ray, depth) the interpolation cell, its four weights, the
//    interpolated continuum, m and T in FP32, and the ray's validity;
//  * k_bin_intensity: one CTA per (ray, chunk of kb bins); a thread owns one sub-bin of two
//    neighbouring bins and walks the depths from the bottom up, holding one intensity pair per
//    direction.  The recurrence needs only the layer optical
//    thicknesses dtau_d = (kappa_d + kappa_{d+1})(m_{d+1} - m_d)/2 and tau_0 = kappa_0 m_0, so
//    no depth array is kept.  The cells and the Planck function of each bin at a window of depths
//    sit in shared memory; the per-bin Planck constants come from the host.
constexpr int kBinThreads = 192;            // at most
constexpr int kBinCols = 2 * kBinThreads;   // sub-bins of a CTA, two per thread
constexpr int kBinMaxKb = 64;

struct DepthCell {
    int r00, dT, dP;        // table row of the lower corner, row offsets to the upper T and P corners
                            // (k_bin_cells); scaled to offsets in pairs of bins for the table
    float w00, w01, w10, w11;
    float m, T, kc;
    float pad[2];
};

struct BinCellArgs {
    int nT, nP, D, n_rays;
    int row_stride;        // bin pairs of a table row
    const double* lt;      // [nT] log10 T axis
    const double* lp;      // [nP] log10 P axis
    const float* kc;       // [nT*nP]
    const double* m;       // [rays][D]
    const double* T;
    const double* P;
    DepthCell* cells;      // [rays][D]
    int* bad;              // [rays], zeroed before the launch
};

struct BinArgs {
    int K, ns, D, n_mu;
    int kb, Dw;            // bins of a CTA (even), depths in shared memory at a time
    const float2* tab;     // [nT*nP][ns][(K + 1) / 2] bin pairs, FP32
    const float3* pk;      // [K]: c1, ln c1, c2 of B_lambda at the bin centre
    const double* w;       // [ns]
    const float* mu;       // [n_mu]
    const DepthCell* cells;
    const int* bad;
    float* out;            // [rays][n_mu][K]
    int* status;           // [rays] or null
};

// index i (0 <= i <= n-2) and fraction f in [0, 1] of x on a strictly increasing axis,
// clamped to its ends (n = 1: i = 0, f = 0)
__device__ __forceinline__ void axis_cell(const double* __restrict__ ax, int n, double x, int* i, double* f) {
    if (n == 1 || x <= ax[0]) { *i = 0; *f = 0.0; return; }
    if (x >= ax[n - 1]) { *i = n - 2; *f = 1.0; return; }
    int lo = 0, hi = n - 1;   // ax[lo] <= x < ax[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (ax[mid] <= x) lo = mid;
        else hi = mid;
    }
    *i = lo;
    *f = (x - ax[lo]) / (ax[lo + 1] - ax[lo]);
}

// A block turns kr rows' chunk of kc bins (even) in shared memory: coalesced reads and writes, at most
// kTabTile values (ns <= 32), eight loads a thread in flight.  by_ns: 2^32 / ns rounded up, so that
// i / ns = umulhi(i, by_ns) for the i < 2^16 here (ns > 1).  57 x 25 x 328 x 12 values: 14.3 us in their
// order, 24.5 turned by blocks that looped over chunks of 64 bins, 16.5 now.
constexpr int kTabTile = 2048;
__global__ void __launch_bounds__(256) k_bin_table(const double* __restrict__ src, float* __restrict__ dst, int rows, int K,
                                                   int ns, unsigned by_ns, int kc, int kr) {
    __shared__ float t[kTabTile + 128];   // [kr][ns][kc + 1]
    const int Kp = (K + 1) & ~1, chunks = (Kp + kc - 1) / kc;
    const int rb = blockIdx.x / chunks, row0 = rb * kr, k0 = (blockIdx.x - rb * chunks) * kc;
    const int nb = min(kc, K - k0), np = min(kc, Kp - k0) >> 1, nr = min(kr, rows - row0);
    const int per = nb * ns, n = nr * per;   // values of a row, of the block (kr = 1 or the whole rows: contiguous)
    const double* in = src + ((size_t)row0 * K + k0) * ns;
    double v[kTabTile / 256];
#pragma unroll
    for (int u = 0; u < kTabTile / 256; ++u) {
        const int i = u * 256 + threadIdx.x;
        v[u] = i < n ? __ldg(in + i) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < kTabTile / 256; ++u) {
        const int i = u * 256 + threadIdx.x;
        if (i >= n) break;
        const int k = ns > 1 ? (int)__umulhi((unsigned)i, by_ns) : i, s = i - k * ns;   // bin over all rows, sub-bin
        const int r = nr > 1 ? k / nb : 0;
        t[(r * ns + s) * (kc + 1) + k - r * nb] = (float)v[u];
    }
    __syncthreads();
    const bool odd = 2 * np > nb;   // the padded bin
    float2* out = reinterpret_cast<float2*>(dst + (size_t)row0 * ns * Kp + k0);
    for (int i = threadIdx.x; i < nr * ns * np; i += 256) {
        const int q = i / np, p = i - q * np;   // q: row and sub-bin
        const float* c = t + q * (kc + 1) + 2 * p;
        out[(size_t)q * (Kp >> 1) + p] = make_float2(c[0], odd && p == np - 1 ? 0.f : c[1]);
    }
}

__global__ void k_bin_cells(BinCellArgs a) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (size_t)a.n_rays * a.D) return;
    const int ray = (int)(i / a.D), d = (int)(i - (size_t)ray * a.D);
    const double md = a.m[i], Td = a.T[i], Pd = a.P[i];
    const bool ok = md > 0.0 && Td > 0.0 && Pd > 0.0 && isfinite(md) && isfinite(Td) && isfinite(Pd) &&
                    (d == 0 || md > a.m[i - 1]);
    if (!ok) atomicOr(a.bad + ray, 1);
    int iT, iP;
    double fT, fP;
    axis_cell(a.lt, a.nT, log10(ok ? Td : 1.0), &iT, &fT);
    axis_cell(a.lp, a.nP, log10(ok ? Pd : 1.0), &iP, &fP);
    DepthCell c;
    c.r00 = iT * a.nP + iP;
    c.dT = (iT + 1 < a.nT ? 1 : 0) * a.nP;
    c.dP = iP + 1 < a.nP ? 1 : 0;
    c.w00 = (float)((1.0 - fT) * (1.0 - fP));
    c.w01 = (float)((1.0 - fT) * fP);
    c.w10 = (float)(fT * (1.0 - fP));
    c.w11 = (float)(fT * fP);
    c.m = (float)md;
    c.T = (float)Td;
    c.kc = c.w00 * a.kc[c.r00] + c.w01 * a.kc[c.r00 + c.dP] + c.w10 * a.kc[c.r00 + c.dT] +
           c.w11 * a.kc[c.r00 + c.dT + c.dP];
    c.pad[0] = c.pad[1] = 0.f;
    c.r00 *= a.row_stride;
    c.dT *= a.row_stride;
    c.dP *= a.row_stride;
    a.cells[i] = c;
}

// Bound by instruction issue (88 % of the slots at one sub-bin per thread): two sub-bins per
// thread in packed FP32.  The two are the same sub-bin of neighbouring bins, and so are a
// warp's: their opacities are alike, where a bin's own sub-bins span orders of magnitude, so a
// warp's layers are mostly all thin or all thick and one of the two forms runs.
// 1024 rays x 80 depths x 328 bins x 12 sub-bins x 5 directions: 1.53 ms one sub-bin per thread,
// 1.37 ms in pairs within a bin, 1.35 ms in pairs across bins, 1.20 ms with the two short forms
// below, 1.17 ms with CTAs of whole warps (bin_chunk).  64 registers and 10 CTAs of three warps per SM.  One
// choice of form for all directions of a layer takes the same time with 93 registers.
// A thread of two sub-bins and all directions is a long chain, and half as many threads share a CTA's
// Planck function.  So a call of few rays spreads its bins and its directions over more CTAs (blockIdx.z
// counts groups of NMU directions), adds threads for the Planck function, and a deep ray keeps a
// window of its depths in shared memory.  Kernel times of one sub-bin per thread, of pairs without and with
// this, in us: one ray of 80 depths, 328 x 12, 5 directions 49, 47, 27; 328 x 1 50, 86, 24; 8 rays of 256
// depths, 16 directions 221, 268, 168; 1024 rays of 200 depths, 328 x 1, 1 direction 565, 1777, 431; 40 x 12,
// 5 directions 213, 249, 167.
template <int NMU>
__global__ void __launch_bounds__(kBinThreads) k_bin_intensity(BinArgs a) {
    extern __shared__ __align__(16) unsigned char bsm[];
    DepthCell* cell = reinterpret_cast<DepthCell*>(bsm);                      // [Dw]
    float* Sb = reinterpret_cast<float*>(cell + a.Dw);                        // [Dw][kb]
    float* part = reinterpret_cast<float*>(bsm);                              // [ns][kb][NMU], after the last depth
    const int ray = blockIdx.y, k0 = blockIdx.x * a.kb, tid = threadIdx.x, D = a.D;
    const int q0 = blockIdx.z * NMU, n_mu = min(NMU, a.n_mu - q0);   // the CTA's directions
    const DepthCell* rc = a.cells + (size_t)ray * D;
    // the window of depths in shared memory: cells and Planck function of the depths w0..top
    int w0;
    auto fill = [&](int top) {
        w0 = max(0, top - a.Dw + 1);
        const int n = top - w0 + 1;
        for (int d = tid; d < n; d += blockDim.x) cell[d] = rc[w0 + d];
        __syncthreads();
        for (int i = tid; i < a.kb * n; i += blockDim.x) {
            const int d = i / a.kb, k = k0 + i - d * a.kb;
            float S = 0.f;
            if (k < a.K) {
                const float3 p = a.pk[k];
                S = planck_f32(p.x, p.y, p.z, cell[d].T);
            }
            Sb[i] = S;
        }
        __syncthreads();
    };
    fill(D - 1);

    const int pairs = a.kb / 2, s = tid / pairs, pr = tid - s * pairs;
    const bool act = s < a.ns && k0 + 2 * pr < a.K;
    const int np = (a.K + 1) >> 1;
    const float2* __restrict__ tab = a.tab + (size_t)s * np + (k0 >> 1) + pr;
    const DepthCell* cw = cell - w0;                                            // depth d: cw[d]
    const float2* Sw = reinterpret_cast<const float2*>(Sb) + pr - w0 * pairs;   // depth d: Sw[d * pairs]
    // a depth's four table values (offsets below 2^31, checked on the host), and its opacity from them
    auto load = [&](int d, float2 (&v)[4]) {
        const int r = cw[d].r00, dT = cw[d].dT, dP = cw[d].dP;
        v[0] = __ldg(tab + r);
        v[1] = __ldg(tab + r + dP);
        v[2] = __ldg(tab + r + dT);
        v[3] = __ldg(tab + r + dT + dP);
    };
    auto kappa = [&](int d, const float2 (&v)[4]) -> float2 {
        const DepthCell& c = cw[d];
        float2 k = ffma2(dup2(c.w00), v[0], dup2(c.kc));
        k = ffma2(dup2(c.w01), v[1], k);
        k = ffma2(dup2(c.w10), v[2], k);
        return ffma2(dup2(c.w11), v[3], k);
    };
    const float2 one = dup2(1.f), minus = dup2(-1.f);
    const float2 nl2 = dup2(-1.4426950408889634f);   // e^{-x} = 2^{x * (-log2 e)}
    float2 I[NMU], mu[NMU], rmu[NMU];                // per direction the intensity, mu and 1/mu
#pragma unroll
    for (int q = 0; q < NMU; ++q) {
        const float m = q < n_mu ? a.mu[q0 + q] : 1.f, r = 1.f / m;
        mu[q] = dup2(m);
        rmu[q] = dup2(r);
        I[q] = make_float2(0.f, 0.f);
    }
    float2 v[4], k_hi, k_lo, dtau, S_hi, Sd;
    if (act) {
        load(D - 1, v);
        k_hi = kappa(D - 1, v);
        load(D - 2, v);
        k_lo = kappa(D - 2, v);
        dtau = fmul2(fadd2(k_lo, k_hi), dup2(0.5f * (cw[D - 1].m - cw[D - 2].m)));
        S_hi = Sw[(D - 1) * pairs], Sd = Sw[(D - 2) * pairs];
        const float2 dS = make_float2((S_hi.x - Sd.x) / dtau.x, (S_hi.y - Sd.y) / dtau.y);
#pragma unroll
        for (int q = 0; q < NMU; ++q) I[q] = ffma2(mu[q], dS, S_hi);
    }
    for (int top = D - 2;;) {
        // the window's layers: d needs the depth below it in the window, but for the last
        const int end = w0 > 0 ? w0 + 1 : 0;
        for (int d = top; act && d >= end; --d) {
            if (d > 0) load(d - 1, v);   // in flight during the layer's directions
            // layer d .. d+1 of optical thickness dtau; per direction x = dtau / mu, e = e^{-x}:
            //   I <- I e + S_d (1 - e) + dS (1 - e(1 + x)) / x,  dS = S_{d+1} - S_d.
            // With B = mu dS / dtau it is S_d + B + e (I - S_{d+1} - B), five operations; its rounding
            // error is the weight's own, 2^-24 dS / x.  Below x = 0.1 instead
            //   I <- I + x (P (S_d - I) + Q dS),  P = (1 - e) / x,  Q = (1 - e(1 + x)) / x^2,
            // P and Q cubics through the four Chebyshev nodes of [0, 0.1] (1.4e-8 and 2.4e-8 off at
            // most, measured on 2001 points with the coefficients as they stand here).
            const float2 dSl = ffma2(Sd, minus, S_hi);
            const float2 G = fmul2(dSl, make_float2(rcp_fast(dtau.x), rcp_fast(dtau.y)));
#pragma unroll
            for (int q = 0; q < NMU; ++q) {
                const float2 x = fmul2(dtau, rmu[q]);
                const bool tx = x.x < 0.1f, ty = x.y < 0.1f;
                float2 r;
                if (!(tx && ty)) {
                    const float2 h = fmul2(x, nl2);
                    const float2 e = make_float2(ex2_fast(h.x), ex2_fast(h.y));
                    const float2 B = fmul2(mu[q], G);
                    r = ffma2(e, ffma2(fadd2(S_hi, B), minus, I[q]), fadd2(Sd, B));
                }
                if (tx || ty) {
                    // (not packed: an instruction's immediate operand holds the coefficient)
                    auto cubic = [](float y, float c3, float c2, float c1, float c0) {
                        return fmaf(y, fmaf(y, fmaf(y, c3, c2), c1), c0);
                    };
                    const float2 P = make_float2(cubic(x.x, -0.04003755832f, 0.1665655674f, -0.4999979837f, 1.f),
                                                 cubic(x.y, -0.04003755832f, 0.1665655674f, -0.4999979837f, 1.f));
                    const float2 Q = make_float2(cubic(x.x, -0.03197662605f, 0.1249158226f, -0.3333316547f, 0.5f),
                                                 cubic(x.y, -0.03197662605f, 0.1249158226f, -0.3333316547f, 0.5f));
                    const float2 t = ffma2(x, ffma2(P, ffma2(I[q], minus, Sd), fmul2(Q, dSl)), I[q]);
                    r = make_float2(tx ? t.x : r.x, ty ? t.y : r.y);
                }
                I[q] = r;
            }
            if (d == 0) break;
            k_hi = k_lo;
            k_lo = kappa(d - 1, v);
            dtau = fmul2(fadd2(k_lo, k_hi), dup2(0.5f * (cw[d].m - cw[d - 1].m)));
            S_hi = Sd;
            Sd = Sw[(d - 1) * pairs];
        }
        if (w0 == 0) break;
        top = w0;
        __syncthreads();
        fill(top);
        cw = cell - w0;
        Sw = reinterpret_cast<const float2*>(Sb) + pr - w0 * pairs;
    }
    const float2 tau0 = fmul2(k_lo, dup2(cw[0].m));
    __syncthreads();   // the window is free for the sub-bins' intensities
    if (act) {
        const float2 ws = dup2((float)a.w[s]);
#pragma unroll
        for (int q = 0; q < NMU; ++q) {
            const float2 h = fmul2(fmul2(tau0, rmu[q]), nl2);
            const float2 e = make_float2(ex2_fast(h.x), ex2_fast(h.y));
            I[q] = fmul2(ws, ffma2(I[q], e, fmul2(Sd, ffma2(e, minus, one))));
            part[(s * a.kb + 2 * pr) * NMU + q] = I[q].x;
            part[(s * a.kb + 2 * pr + 1) * NMU + q] = I[q].y;
        }
    }
    __syncthreads();
    // sum over the sub-bins in order
    const bool bad = a.bad[ray] != 0;
    for (int i = tid; i < a.kb * n_mu; i += blockDim.x) {
        const int b = i / n_mu, q = i - b * n_mu, kk = k0 + b;
        if (kk >= a.K) continue;
        float acc = 0.f;
        for (int t = 0; t < a.ns; ++t) acc += part[(t * a.kb + b) * NMU + q];
        a.out[((size_t)ray * a.n_mu + q0 + q) * a.K + kk] = bad ? __int_as_float(0x7fc00000) : acc;
    }
    if (tid == 0 && a.status && blockIdx.x == 0 && blockIdx.z == 0) a.status[ray] = bad ? 1 : 0;
}

unsigned g_spec_init = 0;

}  // namespace

int formal_launch(int D, int N, const float* kappa, const float* kc, const float* kcont, const float* m, const float* T,
                  double lam0_nm, double lnq, int n_mu, const float* mu, float* I_out, cudaStream_t st) {
    const int blocks = (N + 127) / 128;
    int dev = 0, sms = 0;
    MPSA_CUDA_TRY(cudaGetDevice(&dev));
    MPSA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // One direction per thread while that gives an SM fewer than seven CTAs.  The 80-depth call with one and with
    // five directions per thread: 25,000 points, 5 directions 512 and 517 us, 7 directions 528 and 518; 40,000 points, 2
    // directions 605 and 617, 3 directions 614 and 615, 5 directions 641 and 620; 80,000 points, 2 directions 727 and 731.
    if ((long long)blocks * n_mu >= 7ll * sms)
        k_formal<5><<<dim3(blocks, (n_mu + 4) / 5), 128, 0, st>>>(D, N, kappa, kc, kcont, m, T, lam0_nm, lnq, n_mu, mu, I_out);
    else
        k_formal<1><<<dim3(blocks, n_mu), 128, 0, st>>>(D, N, kappa, kc, kcont, m, T, lam0_nm, lnq, n_mu, mu, I_out);
    MPSA_CUDA_TRY(cudaGetLastError());
    return MPSA_OK;
}

int spectrum_module_init(int device) {
    g_spec_init |= 1u << (device & 31);
    return MPSA_OK;
}

}  // namespace mpsa

using namespace mpsa;

extern "C" int synth_spectrum(mpsa_ctx* ctx, const mpsa_atmos* atm, const mpsa_lgrid* win, int32_t n_mu,
                              const double* mu, float* I_out, const mpsa_synth_opts* opts, void* stream) {
    if (!ctx || !atm || !win || !mu || !I_out) return fail(MPSA_EINVAL, "synth_spectrum: NULL argument");
    if (ctx->L < 1) return fail(MPSA_ESTATE, "synth_spectrum: no line list loaded");
    if (ctx->n_el < 1 || !ctx->d_el) return fail(MPSA_ESTATE, "synth_spectrum: no element table (set_atmosphere_grid)");
    const int D = atm->n_depth;
    if (D < 2 || D > kMaxDepth) return fail(MPSA_EINVAL, "synth_spectrum: n_depth = %d (2..%d)", D, kMaxDepth);
    if (!atm->m || !atm->T || !atm->P) return fail(MPSA_EINVAL, "synth_spectrum: NULL atmosphere array");
    if (atm->comp < 0 || atm->comp >= ctx->n_comp) return fail(MPSA_EINVAL, "synth_spectrum: comp %d", atm->comp);
    if (n_mu < 1 || n_mu > kMaxMu) return fail(MPSA_EINVAL, "synth_spectrum: n_mu = %d (1..%d)", n_mu, kMaxMu);
    for (int q = 0; q < n_mu; ++q)
        if (!(mu[q] > 0 && mu[q] <= 1)) return fail(MPSA_EINVAL, "synth_spectrum: mu[%d] = %g", q, mu[q]);
    for (int d = 0; d < D; ++d) {
        if (!(atm->m[d] > 0) || !(atm->T[d] > 0) || !(atm->P[d] > 0) || !isfinite(atm->m[d]) || !isfinite(atm->T[d]) ||
            !isfinite(atm->P[d]))
            return fail(MPSA_EINVAL, "synth_spectrum: bad depth %d", d);
        if (d > 0 && !(atm->m[d] > atm->m[d - 1])) return fail(MPSA_EINVAL, "synth_spectrum: m not increasing at %d", d);
    }
    int N, r;
    if ((r = check_species(ctx, "synth_spectrum"))) return r;
    if ((r = check_grid(win, &N))) return r;
    if ((size_t)D * ctx->L >= (size_t)1 << 31) return fail(MPSA_EINVAL, "synth_spectrum: n_depth * n_lines >= 2^31");
    MPSA_CUDA_TRY(cudaSetDevice(ctx->device));
    cudaStream_t st = (cudaStream_t)stream;
    Scratch sc(st, ctx->pool);
    const int cont = opts ? opts->continuum : 0;
    const int ne = ctx->n_el;
    // the call's small inputs, in one copy
    std::vector<float> hm(D), hT(D), hmu(n_mu);
    for (int d = 0; d < D; ++d) hm[d] = (float)atm->m[d], hT[d] = (float)atm->T[d];
    for (int q = 0; q < n_mu; ++q) hmu[q] = (float)mu[q];
    HostPack in;
    const size_t oT = in.add(atm->T, D), oP = in.add(atm->P, D), oab = in.add(ctx->h_abund.data() + (size_t)atm->comp * ne, ne);
    const size_t om = in.add(hm.data(), D), of = in.add(hT.data(), D), omu = in.add(hmu.data(), n_mu);
    char* din;
    double* dpop;
    float *kap, *kc, *kcont = nullptr;
    ScratchBlock block;
    block.add(&din, in.data.size());
    block.add(&dpop, (size_t)D * pop_stride(ne));
    block.add(&kap, (size_t)D * N);
    block.add(&kc, D);
    if (cont) block.add(&kcont, (size_t)D * N);
    if ((r = block.take(sc))) return r;
    MPSA_CUDA_TRY(cudaMemcpyAsync(din, in.data.data(), in.data.size(), cudaMemcpyHostToDevice, st));
    const float *fm = reinterpret_cast<float*>(din + om), *fT = reinterpret_cast<float*>(din + of),
                *fmu = reinterpret_cast<float*>(din + omu);
    if ((r = populations_device(ne, ctx->d_el, reinterpret_cast<double*>(din + oab), 1, D, reinterpret_cast<double*>(din + oT),
                                reinterpret_cast<double*>(din + oP), dpop, st)))
        return r;
    if ((r = synth_rows(ctx, dpop, D, nullptr, win->lambda0_nm, win->R, N, kap, kc, nullptr, opts, st))) return r;
    if (cont) {
        if (cont & ~MPSA_CONT_ALL) return fail(MPSA_EINVAL, "synth_spectrum: continuum = %d", cont);
        if ((r = continuum_launch(ctx, dpop, D, nullptr, win->lambda0_nm, win->R, N, cont, kcont, st))) return r;
    }
    if ((r = formal_launch(D, N, kap, kc, kcont, fm, fT, win->lambda0_nm, log1p(1.0 / win->R), n_mu, fmu, I_out, st)))
        return r;
    // pageable host-to-device copies are staged before cudaMemcpyAsync returns,
    // so the host vectors above may go out of scope now
    return MPSA_OK;
}

namespace mpsa {
namespace {

constexpr size_t kBinSmemMax = 227 * 1024;
constexpr int kBinWarps = 8;     // warps of an SM below which directions are shared out over CTAs
constexpr int kPlanckWarps = 24; // warps of an SM below which CTAs take more threads for the Planck function

// Bins of a CTA: an even number up to kBinCols sub-bins.  The warps that the busiest SM is given decide,
// whatever they hold (a quarter of a warp stands for what a CTA costs beside its warps); up to
// eight of them, two per scheduler, take as long as one, and then the spread over the SMs.
int bin_chunk(int K, int ns, long long n_rays, int sms) {
    int best = 2;
    double least = 1e300;
    for (int kb = 2; kb <= kBinMaxKb && kb * ns <= kBinCols; kb += 2) {
        const long long ctas = (K + kb - 1) / kb * n_rays;
        const double load = (double)((ctas + sms - 1) / sms) * ((ns * kb / 2 + 31) / 32 + 0.25);
        const double cost = std::max(load, 8.0) + 0.01 * load;
        if (cost < least) {
            least = cost;
            best = kb;
        }
    }
    return best;
}

template <int NMU>
int bin_launch(BinArgs a, int n_rays, int sms, cudaStream_t st) {
    static unsigned attr_set = 0;   // one bit per device
    static const int regs = [] {
        cudaFuncAttributes fa = {};
        return cudaFuncGetAttributes(&fa, k_bin_intensity<NMU>) == cudaSuccess ? std::max(fa.numRegs, 1) : 128;
    }();
    int dev = 0;
    MPSA_CUDA_TRY(cudaGetDevice(&dev));
    if (!(attr_set & (1u << (dev & 31)))) {
        MPSA_CUDA_TRY(cudaFuncSetAttribute(k_bin_intensity<NMU>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)kBinSmemMax));
        attr_set |= 1u << (dev & 31);
    }
    const dim3 grid((a.K + a.kb - 1) / a.kb, n_rays, (a.n_mu + NMU - 1) / NMU);
    // the threads of the sub-bins, and more for the Planck function while the SMs have few warps
    const long long ctas = (long long)grid.x * grid.y * grid.z;
    int warps = (a.ns * (a.kb / 2) + 31) / 32;
    warps = std::max(warps, (int)std::min<long long>(kBinThreads / 32, kPlanckWarps * sms / ctas));
    // as many depths at a time as leave shared memory for the CTAs that the registers allow
    const int fit = std::max(1, std::min(32, 65536 / (regs * 32 * warps)));
    const size_t per_depth = sizeof(DepthCell) + a.kb * sizeof(float);
    a.Dw = (int)std::min<size_t>(a.D, std::max<size_t>(16, (kBinSmemMax / fit - 1024) / per_depth));
    const size_t smem = std::max(a.Dw * per_depth, (size_t)a.ns * a.kb * NMU * sizeof(float));
    k_bin_intensity<NMU><<<grid, warps * 32, smem, st>>>(a);
    MPSA_CUDA_TRY(cudaGetLastError());
    return MPSA_OK;
}

int check_axis(const double* ax, int n, const char* name) {
    if (n < 1 || !ax) return fail(MPSA_EINVAL, "odf_intensity: %s axis of %d values", name, n);
    for (int i = 0; i < n; ++i) {
        if (!isfinite(ax[i])) return fail(MPSA_EINVAL, "odf_intensity: %s[%d] = %g", name, i, ax[i]);
        if (i > 0 && !(ax[i] > ax[i - 1])) return fail(MPSA_EINVAL, "odf_intensity: %s not increasing at %d", name, i);
    }
    return MPSA_OK;
}

}  // namespace
}  // namespace mpsa

extern "C" int odf_intensity(mpsa_ctx* ctx, const mpsa_odf_table* tab, int32_t n_rays, int32_t n_depth,
                             const double* m, const double* T, const double* P, int32_t n_mu, const double* mu,
                             float* I_out, int32_t* ray_status, void* stream) {
    if (!ctx || !tab || !m || !T || !P || !mu || !I_out) return fail(MPSA_EINVAL, "odf_intensity: NULL argument");
    if (!tab->odf || !tab->kappa_c || !tab->lam_c_nm || !tab->widths)
        return fail(MPSA_EINVAL, "odf_intensity: NULL table array");
    int r;
    if ((r = check_axis(tab->log10_T, tab->nT, "log10_T")) || (r = check_axis(tab->log10_P, tab->nP, "log10_P")))
        return r;
    const int K = tab->K, ns = tab->n_steps;
    if (K < 1) return fail(MPSA_EINVAL, "odf_intensity: K = %d", K);
    if (ns < 1 || ns > 32) return fail(MPSA_EINVAL, "odf_intensity: n_steps = %d (1..32)", ns);
    if ((long long)tab->nT * tab->nP * K * ns >= (1ll << 31))
        return fail(MPSA_EINVAL, "odf_intensity: table of %d x %d x %d x %d", tab->nT, tab->nP, K, ns);
    for (int k = 0; k < K; ++k)
        if (!(tab->lam_c_nm[k] > 0) || !isfinite(tab->lam_c_nm[k]))
            return fail(MPSA_EINVAL, "odf_intensity: lam_c_nm[%d] = %g", k, tab->lam_c_nm[k]);
    double wsum = 0.0;
    for (int s = 0; s < ns; ++s) {
        if (!(tab->widths[s] > 0) || !isfinite(tab->widths[s]))
            return fail(MPSA_EINVAL, "odf_intensity: widths[%d] = %g", s, tab->widths[s]);
        wsum += tab->widths[s];
    }
    if (fabs(wsum - 1.0) > 1e-12) return fail(MPSA_EINVAL, "odf_intensity: widths sum to %.17g", wsum);
    if (n_rays < 1 || n_rays > 65535) return fail(MPSA_EINVAL, "odf_intensity: n_rays = %d (1..65535)", n_rays);
    if (n_depth < 2 || n_depth > kMaxDepth) return fail(MPSA_EINVAL, "odf_intensity: n_depth = %d (2..%d)", n_depth, kMaxDepth);
    if (n_mu < 1 || n_mu > kMaxMu) return fail(MPSA_EINVAL, "odf_intensity: n_mu = %d (1..%d)", n_mu, kMaxMu);
    for (int q = 0; q < n_mu; ++q)
        if (!(mu[q] > 0 && mu[q] <= 1)) return fail(MPSA_EINVAL, "odf_intensity: mu[%d] = %g", q, mu[q]);
    MPSA_CUDA_TRY(cudaSetDevice(ctx->device));
    cudaStream_t st = (cudaStream_t)stream;
    Scratch sc(st, ctx->pool);
    const size_t n_tab = (size_t)tab->nT * tab->nP * ((K + 1) & ~1) * ns, n_cells = (size_t)n_rays * n_depth;
    double *dlt, *dlp, *dw;
    float *dmu, *dtab;
    float3* dpk;
    DepthCell* dcell;
    int* dbad;
    if ((r = sc.alloc(&dlt, tab->nT)) || (r = sc.alloc(&dlp, tab->nP)) || (r = sc.alloc(&dpk, K)) ||
        (r = sc.alloc(&dw, ns)) || (r = sc.alloc(&dmu, n_mu)) || (r = sc.alloc(&dtab, n_tab)) ||
        (r = sc.alloc(&dcell, n_cells)) || (r = sc.alloc(&dbad, n_rays)))
        return r;
    std::vector<float> hmu(n_mu);
    for (int q = 0; q < n_mu; ++q) hmu[q] = (float)mu[q];
    // Planck constants per bin centre: B = c1 / (e^{c2/T} - 1) (FP64 on the host, then FP32)
    std::vector<float3> hpk(K);
    for (int k = 0; k < K; ++k) {
        const double lam_cm = tab->lam_c_nm[k] * 1e-7;
        const double c1 = 2.0 * kH * kC * kC / (lam_cm * lam_cm * lam_cm * lam_cm * lam_cm);
        hpk[k] = make_float3((float)c1, (float)log(c1), (float)(kH * kC / (lam_cm * kKB)));
    }
    MPSA_CUDA_TRY(cudaMemcpyAsync(dlt, tab->log10_T, tab->nT * sizeof(double), cudaMemcpyHostToDevice, st));
    MPSA_CUDA_TRY(cudaMemcpyAsync(dlp, tab->log10_P, tab->nP * sizeof(double), cudaMemcpyHostToDevice, st));
    MPSA_CUDA_TRY(cudaMemcpyAsync(dpk, hpk.data(), K * sizeof(float3), cudaMemcpyHostToDevice, st));
    MPSA_CUDA_TRY(cudaMemcpyAsync(dw, tab->widths, ns * sizeof(double), cudaMemcpyHostToDevice, st));
    MPSA_CUDA_TRY(cudaMemcpyAsync(dmu, hmu.data(), n_mu * sizeof(float), cudaMemcpyHostToDevice, st));
    MPSA_CUDA_TRY(cudaMemsetAsync(dbad, 0, n_rays * sizeof(int), st));
    // whole rows, as many as fit a block, or equal chunks of a row
    const int rows = tab->nT * tab->nP, Kp = (K + 1) & ~1, most = (kTabTile / ns) & ~1, chunks = (Kp + most - 1) / most;
    const int kc = ((Kp + chunks - 1) / chunks + 1) & ~1, kr = chunks > 1 ? 1 : std::max(1, std::min(128 / ns, most / Kp));
    const unsigned by_ns = (unsigned)(((1ull << 32) + ns - 1) / ns);
    k_bin_table<<<(unsigned)((rows + kr - 1) / kr * ((Kp + kc - 1) / kc)), 256, 0, st>>>(tab->odf, dtab, rows, K, ns, by_ns, kc, kr);
    MPSA_CUDA_TRY(cudaGetLastError());
    BinCellArgs ca;
    ca.nT = tab->nT;
    ca.nP = tab->nP;
    ca.D = n_depth;
    ca.n_rays = n_rays;
    ca.row_stride = (K + 1) / 2 * ns;
    ca.lt = dlt;
    ca.lp = dlp;
    ca.kc = tab->kappa_c;
    ca.m = m;
    ca.T = T;
    ca.P = P;
    ca.cells = dcell;
    ca.bad = dbad;
    k_bin_cells<<<(unsigned)((n_cells + 255) / 256), 256, 0, st>>>(ca);
    MPSA_CUDA_TRY(cudaGetLastError());
    BinArgs a;
    a.K = K;
    a.ns = ns;
    a.D = n_depth;
    a.n_mu = n_mu;
    a.tab = reinterpret_cast<const float2*>(dtab);
    a.pk = dpk;
    a.w = dw;
    a.mu = dmu;
    a.cells = dcell;
    a.bad = dbad;
    a.out = I_out;
    a.status = ray_status;
    prof_mark(ctx, MPSA_KERNEL_BINS, st);
    int dev = 0, sms = 0;
    MPSA_CUDA_TRY(cudaGetDevice(&dev));
    MPSA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // directions of a thread: all (in two groups above eight, which take 135 registers at once), or fewer
    // while that leaves an SM no more than kBinWarps warps
    int nq = 1;
    for (; nq < n_mu; ++nq) {
        const int z = (n_mu + nq - 1) / nq;
        a.kb = bin_chunk(K, ns, (long long)n_rays * z, sms);
        if ((long long)((K + a.kb - 1) / a.kb) * n_rays * z * ((ns * a.kb / 2 + 31) / 32) <= kBinWarps * sms) break;
    }
    if (nq > 8) nq = (n_mu + 1) / 2;
    a.kb = bin_chunk(K, ns, (long long)n_rays * ((n_mu + nq - 1) / nq), sms);
    switch (nq) {
        case 1: r = bin_launch<1>(a, n_rays, sms, st); break;
        case 2: r = bin_launch<2>(a, n_rays, sms, st); break;
        case 3: r = bin_launch<3>(a, n_rays, sms, st); break;
        case 4: r = bin_launch<4>(a, n_rays, sms, st); break;
        case 5: r = bin_launch<5>(a, n_rays, sms, st); break;
        case 6: r = bin_launch<6>(a, n_rays, sms, st); break;
        case 7: r = bin_launch<7>(a, n_rays, sms, st); break;
        default: r = bin_launch<8>(a, n_rays, sms, st); break;
    }
    prof_mark(ctx, MPSA_KERNEL_BINS, st);
    // pageable host-to-device copies are staged before cudaMemcpyAsync returns,
    // so the host vectors above may go out of scope now
    return r;
}
