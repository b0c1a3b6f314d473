// synth_opacity: line-by-line opacity on a log-lambda grid.
//
// Paper: Eq. (l_nu_line) of Sect. 2.1 summed over every line of the list on
// the grid lambda_j = lambda_0 (1 + 1/R)^j of App. E, with the cut of Sect. 4.3 /
// App. E (a line contributes where its absorption coefficient is at least
// cut * kappa_c; kappa_c is the flat continuum kc_factor * median line-centre
// opacity of the synthetic workload).
//
// Pipeline (all on the caller's stream):
//   k_start        per line: how far off the grid its centre is; per (row, species):
//                  ln(sqrt(pi) e^2/(m_e c) N/U / rho), u, c/u from the FP64 table
//   k_kappa0       per (row, line): ln S, a, ln kappa0 in FP32 log space; on long lists and narrow
//                  grids k_bounds instead: upper bounds of ln kappa0 and ln(a S)
//   k_med_*        per row: lower median of ln kappa0 -> ln t_p, kappa_c
//   k_prep         per (row, line): peak against the cut, reach of the wing; the lines left, listed
//   k_place        the listed lines' centre index c and fraction f on the grid (FP64 log)
//   k_windows      per listed line: its terms where there are only bounds so far; cut windows (outer: no
//                  point beyond can pass the cut; inner: every point inside passes), width class
//   k_scan_class, k_scatter   stable counting sort of the kept lines by width class
//   k_ranges       per (row, class, tile boundary): first line whose centre lies at or
//                  beyond the boundary (binary search in the centre-sorted class)
//   k_tiles        the profile kernel: one CTA per (row, tile of 2048 or 4096 points), or several on
//                  calls with few tiles; wings summed at Chebyshev nodes, the rest point by point; FP32
//                  partial sums folded into Kahan-compensated totals; no atomics; coalesced stores.
#include <math.h>
#include <stdio.h>

#include <algorithm>
#include <vector>

#include "common.cuh"
#include "voigt.cuh"
#include "internal.cuh"

namespace mpsa {

namespace {

constexpr float kLn10 = 2.302585092994046f;
constexpr float kFourPi = 12.566370614359172f;

__device__ __forceinline__ int floordiv(int a, int b) { return (a >= 0) ? a / b : -((-a + b - 1) / b); }

// A wavelength grid as the preparation kernels see it: lambda_j = lam0 e^{j lnq}, N points, the
// index of its per-line arrays (distance, flags, placement).
struct GridDesc {
    double lam0_nm, lnq64;
    float lnq, inv_first, inv_last;   // ln q and 1/lambda of the first and last point [1/nm]
    int N, index;
};
// The grid of each row: one for all rows, or grids[row].
struct RowGrids {
    GridDesc one;
    const GridDesc* many;
    __device__ __forceinline__ GridDesc of(int s) const { return many ? many[s] : one; }
};
// Where the rows' continuum and evaluation counts go (either may be null): one array for all
// rows, or a pointer per row.
struct RowOut {
    float* kc;
    unsigned long long* ev;
    float* const* kc_many;
    unsigned long long* const* ev_many;
    __device__ __forceinline__ float* kc_of(int s) const { return kc_many ? kc_many[s] : (kc ? kc + s : nullptr); }
    __device__ __forceinline__ unsigned long long* ev_of(int s) const {
        return ev_many ? ev_many[s] : (ev ? ev + s : nullptr);
    }
};

// k_place: c = floor(x0), f = x0 - c with x0 = ln(lambda0/lambda_start)/ln(1+1/R) (FP64: an FP32
// logarithm would misplace lines by whole grid points) of the lines that some row of the
// grid keeps.  A CTA gathers the kept ones of its 1024 lines and then takes their logarithms
// with full warps: FP64 bounds this kernel, and of a 5e6-line list a window of a few nm keeps a
// few per cent (all 5e6: 484 us, 104 us for the 3 per cent that 80 depths keep of a 7 nm window).
// LINES: 1024, or 256 for lists too short to give every SM a CTA of 1024.
template <int LINES>
__global__ void __launch_bounds__(kPrepThreads) k_place(int64_t L, size_t ld, const double* __restrict__ lam_nm, GridDesc one,
                                                        const GridDesc* __restrict__ many,
                                                        const unsigned char* __restrict__ flag, int* __restrict__ c_out,
                                                        float* __restrict__ f_out) {
    __shared__ short list[LINES];
    __shared__ int n_list;
    const int g = blockIdx.y, tid = threadIdx.x, lane = tid & 31;
    const int64_t i0 = (int64_t)blockIdx.x * LINES;
    if (tid == 0) n_list = 0;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < LINES / kPrepThreads; ++k) {
        const int off = k * kPrepThreads + tid;
        const bool on = i0 + off < L && flag[g * ld + i0 + off] != 0;
        const unsigned m = __ballot_sync(0xffffffffu, on);
        int base = 0;
        if (lane == 0 && m) base = atomicAdd(&n_list, __popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (on) list[base + __popc(m & ((1u << lane) - 1u))] = (short)off;
    }
    __syncthreads();
    const GridDesc q = many ? many[g] : one;
    for (int t = tid; t < n_list; t += kPrepThreads) {
        const int64_t i = i0 + list[t];
        double x0 = log(lam_nm[i] / q.lam0_nm) / q.lnq64;
        x0 = fmin(fmax(x0, -268435456.0), 268435456.0);
        const double c = floor(x0);
        c_out[g * ld + i] = (int)c;
        f_out[g * ld + i] = (float)(x0 - c);
    }
}

// per-row scalars (FP32) and per-(row, species) scalars
struct RowConst {
    float ne, nHI, inv_kT_eV, hc_kT_cm;
};
struct __align__(16) SpConst {
    float lnC, u, kv, lnu;   // lnu = logf(u)
};

__device__ __forceinline__ void sp_consts(int t, const int* __restrict__ sel, int n_sp, const int* __restrict__ sp_el,
                                          const int* __restrict__ sp_stage, int n_el, const double* __restrict__ el,
                                          const double* __restrict__ pop, double vturb, int pop32,
                                          RowConst* __restrict__ rc, SpConst* __restrict__ sc) {
    const int s = t / n_sp, sp = t % n_sp;
    const double* row = pop + (size_t)(sel ? sel[s] : s) * pop_stride(n_el);
    const double T = row[kPopT];
    const int e = sp_el[sp], st = sp_stage[sp];
    const double m = el[e * kElStride + kElMass] * kAMU;
    const double u = sqrt(2.0 * kKB * T / m + vturb * vturb);
    const double NU = row[pop_nu(e, st)];
    const double pre = sqrt(kPI) * kE * kE / (kME * kC);
    SpConst o;
    if (pop32)   // precision-study variant: the population table rounded to FP32 first
        o.lnC = NU > 0 ? (float)log(pre) + logf((float)NU) - logf((float)row[kPopRho]) : -INFINITY;
    else
        o.lnC = NU > 0 ? (float)(log(pre) + log(NU) - log(row[kPopRho])) : -INFINITY;
    o.u = (float)u;
    o.kv = (float)(kC / u);
    o.lnu = logf(o.u);
    sc[t] = o;
    if (sp == 0) {
        RowConst r;
        r.ne = (float)row[kPopNe];
        r.nHI = (float)row[kPopNHI];
        r.inv_kT_eV = (float)(kEV / (kKB * T));
        r.hc_kT_cm = (float)(kH * kC / (kKB * T));
        rc[s] = r;
    }
}

// k_start: two independent tables, by blocks of one launch.
// The first `cb` blocks: the constants of each (row, species), and the rows' counts of listed
// lines set to zero.
// The others: per (grid, line), a lower bound of the distance between a centre off the grid and
// the grid's nearest point in relative frequency, |v| / kv there:
//   1 - lambda/lambda_0 (centre shortward), lambda/lambda_{N-1} - 1 (longward),
// negative for centres on the grid.  Four grid points and the FP32 rounding are taken off, so FP32 will do, and no
// logarithm is needed: the exact position of a line (k_place) is formed only if it reaches the
// grid.  Clears the line's flag.
constexpr int kStartThreads = 128;
__global__ void __launch_bounds__(kStartThreads) k_start(int cb, int n_sel, const int* __restrict__ sel, int n_sp,
                                                         const int* __restrict__ sp_el, const int* __restrict__ sp_stage,
                                                         int n_el, const double* __restrict__ el,
                                                         const double* __restrict__ pop, double vturb, int pop32,
                                                         RowConst* __restrict__ rc, SpConst* __restrict__ sc,
                                                         int* __restrict__ nsurv, int64_t L, size_t ld, int n_grids,
                                                         const double* __restrict__ lam_nm, GridDesc one,
                                                         const GridDesc* __restrict__ many, float* __restrict__ dist,
                                                         unsigned char* __restrict__ flag) {
    if ((int)blockIdx.x < cb) {
        const int t = blockIdx.x * kStartThreads + threadIdx.x;
        if (t < n_sel) nsurv[t] = 0;
        if (t < n_sel * n_sp) sp_consts(t, sel, n_sp, sp_el, sp_stage, n_el, el, pop, vturb, pop32, rc, sc);
        return;
    }
    const int64_t i = (int64_t)(blockIdx.x - cb) * kStartThreads + threadIdx.x;
    if (i >= L) return;
    const float lam = (float)lam_nm[i];
    for (int g = 0; g < n_grids; ++g) {
        const GridDesc q = many ? many[g] : one;
        const float d = fmaxf(fmaf(-lam, q.inv_first, 1.f), fmaf(lam, q.inv_last, -1.f));
        // lambda, 1/lambda_0 and the product round by 6e-8 each
        dist[g * ld + i] = fmaf(d, 1.f - 4.2f * q.lnq - 1e-5f, -4.2f * q.lnq - 4e-7f);
        flag[g * ld + i] = 0;
    }
}

// ---------------------------------------------------------------------------
// k_kappa0: Eq. (l_nu_line) in log space, FP32.
//   Delta nu_D = u / lambda0, a = gamma / (4 pi Delta nu_D),
//   ln S = ln C_s + ln(gf) - E/kT + ln(1 - e^{-h nu0/kT}) - ln Delta nu_D,
//   ln kappa0 = ln S + ln H(0, a).
// One thread per line and up to kKappa0Rows rows: the line's data and its three damping
// constants are read and formed once, then each row's values follow.
//
// H(0, a) is bound by its arithmetic: at v = 0 the two poles of a pair of voigt_core give the same
// term, so voigt_core0 forms it once (60 operations instead of 130), with every rounding that the general
// form takes there (median, cut and windows follow from these bits).  4e8 (row, line) pairs: 3.60 ms
// in the general form, 2.58 ms; their 12 bytes each would take 0.7 ms (k_bounds below avoids most of it).
constexpr int kKappa0Rows = 16;

__device__ __forceinline__ float voigt_core0(float a) {
    const float d = kGHDelta, Y1 = __fadd_rn(a, d);
    float sum = 0.f;
    if (a < 2.f) {
        const float Yd = __fadd_rn(Y1, d);
#pragma unroll
        for (int k = 0; k < kGHPairs; ++k) {
            const float sk = c_voigt.s[k], s2 = __fmul_rn(sk, sk);
            const float p = __fmul_rn(__fadd_rn(s2, d * d), __fmaf_rn(Y1, Y1, s2));
            const float t = __fmaf_rn(c_voigt.U[k], __fmaf_rn(-Y1, d, s2), __fmul_rn(__fmul_rn(c_voigt.S[k], -sk), Yd));
            sum = __fmaf_rn(__fmaf_rn(t, p, __fmul_rn(t, p)), rcp_approx(__fmul_rn(p, p)), sum);
        }
        return __fmaf_rn(a, sum, 1.f);
    }
    const float Y12 = __fmul_rn(Y1, Y1);
#pragma unroll
    for (int k = 0; k < kGHPairs; ++k) {
        const float sk = c_voigt.s[k];
        const float q = __fmaf_rn(sk, sk, Y12), g = __fmaf_rn(c_voigt.S[k], sk, __fmul_rn(c_voigt.U[k], Y1));
        sum = __fmaf_rn(__fmaf_rn(q, g, __fmul_rn(q, g)), rcp_approx(__fmul_rn(q, q)), sum);
    }
    return sum;
}

// order-preserving keys of the FP32 bit patterns
__device__ __forceinline__ unsigned fkey(float x) {
    unsigned b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float unkey(unsigned k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// Where the median of a row is looked for (see the median below).
struct MedState {
    unsigned lo, hi;   // keys that bracket it
    unsigned below;    // lines below lo
    unsigned n;        // lines in the bracket, listed
};

// The line list, and one line's parameters with what does not depend on the row.
struct LineList {
    const int* species;
    const float *loggf, *E, *lgR, *lgS, *lgW;
    const double* lam_nm;
};
struct LineConst {
    float lam, lglam, lg, E, gR, gS, gW;
};
__device__ __forceinline__ LineConst line_const(const LineList& l, int64_t i) {
    const float lam = (float)(l.lam_nm[i] * 1e-7);
    return LineConst{lam, logf(lam), l.loggf[i], l.E[i], exp10f(l.lgR[i]), exp10f(l.lgS[i]), exp10f(l.lgW[i])};
}
// ln kappa0, ln S and a of a line in a row.  Every kernel that forms them takes the same roundings
// (the fused operations are spelled out), so a line has one value wherever it is formed.
__device__ __forceinline__ float line_terms(const LineConst& l, const RowConst& r, const SpConst& q, float* lnS, float* a) {
    const float gamma = __fmaf_rn(l.gW, r.nHI, __fmaf_rn(l.gS, r.ne, l.gR));
    *a = __fmul_rn(gamma, l.lam) / __fmul_rn(kFourPi, q.u);
    const float stim = -expm1f(-r.hc_kT_cm / l.lam);
    const float t = __fmaf_rn(-l.E, r.inv_kT_eV, __fmaf_rn(l.lg, kLn10, q.lnC));
    *lnS = __fsub_rn(__fadd_rn(t, logf(stim)), __fsub_rn(q.lnu, l.lglam));
    return __fadd_rn(*lnS, logf(*a * *a >= 36.f ? voigt_H(0.f, *a) : voigt_core0(*a)));
}

// SAMPLE: every kMedStride-th line only, ln kappa0 alone, into lnk0_out [n_sel][ld].
constexpr int kMedStride = 128;
template <bool SAMPLE>
__global__ void k_kappa0(int64_t L, size_t ld, int n_sel, LineList lines, int n_sp, const RowConst* __restrict__ rc,
                         const SpConst* __restrict__ sc, float* __restrict__ lnS_out, float* __restrict__ a_out,
                         float* __restrict__ lnk0_out) {
    const int64_t at = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, i = SAMPLE ? at * kMedStride : at;
    if (i >= L) return;
    const int sp = lines.species[i];
    const LineConst l = line_const(lines, i);
    const int s1 = min(n_sel, (int)(blockIdx.y + 1) * kKappa0Rows);
#pragma unroll 1
    for (int s = blockIdx.y * kKappa0Rows; s < s1; ++s) {
        const size_t o = s * ld + at;
        float lnS, a;
        lnk0_out[o] = line_terms(l, rc[s], sc[(size_t)s * n_sp + sp], &lnS, &a);
        if (!SAMPLE) {
            lnS_out[o] = lnS;
            a_out[o] = a;
        }
    }
}

// k_bounds: upper bounds of ln kappa0 and of ln(a S) of every (row, line), for long lists.
// Of such a list a window keeps some per cent, and the median needs the few per cent around it, so
// only those take the full terms (k_med_collect, k_windows); the rest is sorted out by bounds
// that cost a tenth: ln(1 - e^-x) through ex2/lg2 (x itself below 0.02, at most 1 per cent
// more), and H(0, a) = e^{a^2} erfc(a) <= 2/(sqrt(pi) (a + sqrt(a^2 + 4/pi))) (Abramowitz & Stegun
// 7.1.13), at most 0.057 in the logarithm above it for any a.  kBoundUp lies above the roundings of
// both forms; ln kappa0 is above its bound less kBoundGap.  Both grow with the magnitude, for
// lists whose terms leave the usual range.
// 4e8 pairs: 2.58 ms for the full terms, 0.74 ms for the bounds, 8 bytes each.
constexpr float kBoundUp = 0.02f, kBoundGap = 0.12f, kBoundRel = 1e-6f;
__device__ __forceinline__ float lg2_fast(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float ex2_fast(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float sqrt_fast(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// up by the margin; an infinity stays what it is
__device__ __forceinline__ float bound_up(float x) { return x + fmaf(kBoundRel, fminf(fabsf(x), 1e30f), kBoundUp); }
// a value that ln kappa0 is not below, from its upper bound
__device__ __forceinline__ float bound_low(float up) { return up - fmaf(3.f * kBoundRel, fminf(fabsf(up), 1e30f), kBoundGap); }

__global__ void __launch_bounds__(256) k_bounds(int64_t L, size_t ld, int n_sel, LineList lines, int n_sp,
                                                const RowConst* __restrict__ rc, const SpConst* __restrict__ sc,
                                                float* __restrict__ lnaS_up, float* __restrict__ lnk0_up) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L) return;
    constexpr float kLn2 = 0.6931471805599453f, kLog2E = 1.4426950408889634f;
    const int sp = lines.species[i];
    const LineConst l = line_const(lines, i);
    const float lgk = fmaf(l.lg, kLn10, l.lglam), inv = kLog2E / l.lam;
    const float da = l.lam * (float)(1.0 / (4.0 * kPI * kC));   // a = gamma lambda kv / (4 pi c), kv = c / u
    const int s1 = min(n_sel, (int)(blockIdx.y + 1) * kKappa0Rows);
#pragma unroll 2
    for (int s = blockIdx.y * kKappa0Rows; s < s1; ++s) {
        const RowConst r = rc[s];
        const SpConst q = sc[(size_t)s * n_sp + sp];
        const float a = fmaf(l.gW, r.nHI, fmaf(l.gS, r.ne, l.gR)) * (da * q.kv);
        const float x2 = r.hc_kT_cm * inv;   // x log2(e)
        const float w = x2 < 0.02f * kLog2E ? x2 * kLn2 : 1.f - ex2_fast(-x2);
        const float lnS = fmaf(kLn2, lg2_fast(w), fmaf(-l.E, r.inv_kT_eV, (q.lnC - q.lnu) + lgk));
        float k0 = fmaf(-kLn2, lg2_fast(a + sqrt_fast(fmaf(a, a, 1.2732395f))), lnS + 0.1207822f);   // ln(2/sqrt(pi))
        if (!(a < 1.0e18f)) k0 = __int_as_float(0x7fc00000);   // a^2 beyond FP32: no bound, the line takes its full terms
        const size_t o = s * ld + i;
        lnaS_up[o] = bound_up(fmaf(kLn2, lg2_fast(a), lnS));
        lnk0_up[o] = bound_up(k0);
    }
}

// ---------------------------------------------------------------------------
// Lower median (rank (L-1)/2) of ln kappa0 per row, exact, on the order-preserving keys.
//
// Lists of up to kMedSmall lines: one CTA per row selects it in three radix levels of 11, 11 and 10
// bits (k_med_select).  Longer ones are read once instead of three times: every 128th line is formed
// ahead, two order statistics of that sample bracket the median (k_med_bracket: five standard
// deviations of its rank on either side), one pass over the row counts the lines below the bracket
// and lists the 3 per cent inside (k_med_collect), and the median is selected among those
// (k_med_select again; from the whole row should the bracket have missed it).  5e6 lines x 80
// rows: 1.10 ms for three passes, 0.62 ms over stored values, 0.80 ms over bounds of them (which save
// 1.85 ms in k_kappa0).  (Counting and listing in k_kappa0 itself took one global atomic per warp
// and row: 2.6 -> 11.5 ms.)
constexpr int kMedBins = 2048, kMedThreads = 1024;
constexpr int64_t kMedSmall = 65536;

// The key of rank `rank` among the keys key(x[0..n)), x 16-byte aligned: all threads of the CTA
// call it.
template <class F>
__device__ __forceinline__ unsigned block_select(const float* __restrict__ x, int64_t n, unsigned rank, unsigned* h,
                                                 F&& key) {
    __shared__ unsigned wsum[32];
    __shared__ unsigned s_bin, s_rank;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned prefix = 0u;
    for (int level = 0; level < 3; ++level) {
        const int shift = level == 0 ? 21 : (level == 1 ? 10 : 0), nb = level == 2 ? 1024 : 2048;
        const unsigned pmask = level == 0 ? 0u : (0xffffffffu << (level == 1 ? 21 : 10));
        for (int i = tid; i < kMedBins; i += kMedThreads) h[i] = 0u;
        __syncthreads();
        auto add = [&](float v) {
            const unsigned k = key(v);
            if ((k & pmask) == prefix) atomicAdd(&h[(k >> shift) & (nb - 1)], 1u);
        };
        const int64_t n4 = n >> 2;
#pragma unroll 4
        for (int64_t i = tid; i < n4; i += kMedThreads) {
            const float4 q = __ldg(reinterpret_cast<const float4*>(x) + i);
            add(q.x), add(q.y), add(q.z), add(q.w);
        }
        if (tid < (int)(n & 3)) add(__ldg(x + 4 * n4 + tid));
        __syncthreads();
        // two bins per thread; block-wide inclusive scan of their counts
        const unsigned c0 = h[2 * tid], c1 = h[2 * tid + 1], v = c0 + c1;
        unsigned incl = v;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += y;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        unsigned before = incl - v;
        for (int w = 0; w < warp; ++w) before += wsum[w];
        if (rank >= before && rank < before + v) {   // one thread
            const bool low = rank < before + c0;
            s_bin = 2u * tid + (low ? 0u : 1u);
            s_rank = rank - (low ? before : before + c0);
        }
        __syncthreads();
        prefix |= s_bin << shift;
        rank = s_rank;
        __syncthreads();
    }
    return prefix;
}

// sample [n_sel][ld] of n values: keys around the middle, wide enough for the median of the whole
__global__ void __launch_bounds__(kMedThreads) k_med_bracket(int64_t n, size_t ld, const float* __restrict__ sample,
                                                             MedState* __restrict__ st) {
    __shared__ unsigned h[kMedBins];
    const int s = blockIdx.x;
    const float* x = sample + s * ld;
    const int64_t mid = (n - 1) / 2, w = (int64_t)(2.5 * sqrt((double)n)) + 2;
    const unsigned lo = block_select(x, n, (unsigned)(mid - w < 0 ? 0 : mid - w), h, [](float v) { return fkey(v); });
    const unsigned hi = block_select(x, n, (unsigned)(mid + w >= n ? n - 1 : mid + w), h, [](float v) { return fkey(v); });
    if (threadIdx.x == 0) st[s] = MedState{lo, hi, 0u, 0u};
}

// Count the row's lines below its bracket, list those inside (list [n_sel][list_ld], any order).
// The row holds upper bounds: the lines that these leave open go to the warp's queue, and take
// their full terms 32 at a time.  (A queue per CTA of 1024 threads, 1.51 ms for 5e6 lines x 80 rows, waited at
// its barriers; 0.68 ms now.)
constexpr int kCollectThreads = 256;
__global__ void __launch_bounds__(kCollectThreads) k_med_collect(int64_t L, size_t ld, const float* __restrict__ lnk0_up,
                                                                 LineList lines, int n_sp, const RowConst* __restrict__ rc,
                                                                 const SpConst* __restrict__ sc, MedState* __restrict__ st,
                                                                 float* __restrict__ list, size_t list_ld) {
    constexpr int kWarps = kCollectThreads / 32;
    __shared__ int queue[kWarps][32 + 128];
    const int s = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lo = st[s].lo, hi = st[s].hi, lt = (1u << lane) - 1u;
    const float flo = unkey(lo), fhi = unkey(hi);
    const float* x = lnk0_up + s * ld;   // rows 16-byte aligned and padded to four lines
    const RowConst r = rc[s];
    int* const q = queue[warp];
    int nq = 0;
    unsigned below = 0u;
    auto take = [&](int n) {   // the queue's last n lines
        nq -= n;
        bool in = false;
        float v = 0.f;
        if (lane < n) {
            const int64_t i = q[nq + lane];
            float lnS, a;
            v = line_terms(line_const(lines, i), r, sc[(size_t)s * n_sp + lines.species[i]], &lnS, &a);
            const unsigned k = fkey(v);
            below += k < lo;
            in = k >= lo && k <= hi;
        }
        const unsigned m = __ballot_sync(0xffffffffu, in);
        unsigned at = 0u;
        if (lane == 0 && m) at = atomicAdd(&st[s].n, (unsigned)__popc(m));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (in) list[s * list_ld + at + __popc(m & lt)] = v;
        __syncwarp();
    };
    const int64_t step = (int64_t)gridDim.x * kWarps * 128;
    int64_t i0 = ((int64_t)blockIdx.x * kWarps + warp) * 128;
    auto load = [&](int64_t j) {
        return j + 4 * lane < L ? __ldg(reinterpret_cast<const float4*>(x + j) + lane) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    float4 next = load(i0);
    for (; i0 < L; i0 += step) {
        const float4 f = next;
        next = load(i0 + step);
        const float v[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int64_t i = i0 + 4 * lane + c;
            const bool on = i < L, under = v[c] < flo;
            below += on && under;
            const bool open = on && !under && !(bound_low(v[c]) > fhi);
            const unsigned m = __ballot_sync(0xffffffffu, open);
            if (open) q[nq + __popc(m & lt)] = (int)i;
            nq += __popc(m);
        }
        __syncwarp();
        while (nq >= 32) take(32);
    }
    if (nq > 0) take(nq);
    below = __reduce_add_sync(0xffffffffu, below);
    if (lane == 0 && below) atomicAdd(&st[s].below, below);
}

// whether the median lies in the row's bracket
__device__ __forceinline__ bool med_found(const MedState& m, int64_t L) {
    const unsigned rank = (unsigned)((L - 1) / 2);
    return rank >= m.below && rank - m.below < m.n;
}

// ln kappa0 in place of its bound, for the rows whose bracket missed the median
__global__ void __launch_bounds__(256) k_med_redo(int64_t L, size_t ld, LineList lines, int n_sp,
                                                  const RowConst* __restrict__ rc, const SpConst* __restrict__ sc,
                                                  const MedState* __restrict__ st, float* __restrict__ lnk0) {
    const int s = blockIdx.y;
    if (med_found(st[s], L)) return;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < L; i += (int64_t)gridDim.x * blockDim.x) {
        float lnS, a;
        lnk0[s * ld + i] = line_terms(line_const(lines, i), rc[s], sc[(size_t)s * n_sp + lines.species[i]], &lnS, &a);
    }
}

// st: null, or the bracket whose lines are listed
__global__ void __launch_bounds__(kMedThreads) k_med_select(int64_t L, size_t ld, const float* __restrict__ lnk0,
                                                            const MedState* __restrict__ st,
                                                            const float* __restrict__ list, size_t list_ld,
                                                            float ln_kc_factor, float ln_cut, float* __restrict__ ln_tp,
                                                            RowOut out) {
    __shared__ unsigned h[kMedBins];
    const int s = blockIdx.x;
    const float* x = lnk0 + s * ld;
    int64_t n = L;
    unsigned rank = (unsigned)((L - 1) / 2), lo = 0u;
    int sh = 0;
    if (st && med_found(st[s], L)) {
        x = list + s * list_ld;
        n = st[s].n;
        rank -= st[s].below;
        // listed keys differ in their low bits only: spread them over the bins
        lo = st[s].lo;
        sh = __clz((int)((st[s].hi - lo) | 1u));
    }
    const float med = unkey(lo + (block_select(x, n, rank, h, [&](float v) { return (fkey(v) - lo) << sh; }) >> sh));
    if (threadIdx.x == 0) {
        ln_tp[s] = med + ln_kc_factor + ln_cut;
        float* const kc = out.kc_of(s);
        if (kc) *kc = expf(med + ln_kc_factor);
    }
}

// ---------------------------------------------------------------------------
// Cut windows.  For H monotone in |v| the points where s_rel * H(v, a) >= 1 form
// |v| <= v*.  Bisection (geometric, 40 steps) on the FP32 H gives
//   v_out: H(v) < r (1 - 1e-4) for all v >= v_out  (no point beyond can pass the cut)
//   v_in : H(v) >= r (1 + 1e-4) for all v <= v_in  (every point inside passes)
// with r = 1/s_rel; the margins exceed the FP32 errors of H (3e-6) and of v (2e-6).
// H(v, a) <= 4a/(sqrt(pi) v^2) + exp(-v^2/4) bounds the search.
__device__ float v_bound(float a, float t) {
    return fmaxf(sqrtf(8.f * a * kInvSqrtPi / t), 2.f * sqrtf(logf(fmaxf(2.f / t, 1.f)))) * 1.01f + 1.f;
}

// Crossing of H(v, a) = t by the Illinois variant of regula falsi on ln H against ln v.
// Invariant: H(e^xlo) >= t > H(e^xhi); the bracket shrinks to a few FP32 ulps of ln v.
// The search first tries a bracket of +-5 % around ve = max(sqrt(a / (sqrt(pi) t)),
// sqrt(-ln t)), the crossing of the Lorentz wing a / (sqrt(pi) v^2) or of the Doppler core
// e^{-v^2}; where H confirms it the search starts there, else from the ends it has verified.
// Returns the verified ends.
__device__ void crossing(float a, float t, float vb, float* v_ge, float* v_lt) {
    const float lt = logf(t);
    auto f = [&](float x) {
        const float h = voigt_H(expf(x), a);
        return h > 0.f ? logf(h) - lt : -1.0e4f;
    };
    float xlo = logf(1e-4f), xhi = logf(vb), flo, fhi;
    const float ve = fmaxf(sqrtf(a * kInvSqrtPi / t), sqrtf(fmaxf(-lt, 0.f)));
    const float xg0 = logf(ve) - 0.05f, xg1 = xg0 + 0.1f;
    bool probe_lo = true;
    if (xg0 > xlo && xg1 < xhi) {
        const float f0 = f(xg0);
        if (f0 >= 0.f) {                   // H >= t at xg0, so also at |v| = 1e-4
            probe_lo = false;
            xlo = xg0;
            flo = f0;
            const float f1 = f(xg1);
            if (f1 < 0.f) {
                xhi = xg1;
                fhi = f1;
            } else {
                xlo = xg1;
                flo = f1;
                fhi = f(xhi);
            }
        } else {
            xhi = xg0;
            fhi = f0;
        }
    } else {
        fhi = f(xhi);
    }
    if (probe_lo) {
        flo = f(xlo);
        if (flo < 0.f) {                   // below t already at |v| = 1e-4
            *v_ge = -1.f;
            *v_lt = 1e-4f;
            return;
        }
    }
    int side = 0;
    // stop at ~2 FP32 ulps of ln v (the ends stay verified, so precision only sets tightness)
    for (int it = 0; it < 60 && xhi - xlo > 3e-7f * fmaxf(1.f, fabsf(xhi)); ++it) {
        float x = (xlo * fhi - xhi * flo) / (fhi - flo);
        if (!(x > xlo && x < xhi)) x = 0.5f * (xlo + xhi);
        if (!(x > xlo && x < xhi)) break;
        const float fx = f(x);
        if (fx >= 0.f) {
            xlo = x;
            flo = fx;
            if (side == 1) fhi *= 0.5f;
            side = 1;
        } else {
            xhi = x;
            fhi = fx;
            if (side == -1) flo *= 0.5f;
            side = -1;
        }
    }
    *v_ge = expf(xlo);
    *v_lt = expf(xhi);
}

// The inner speed lies just inside the outer crossing: where H falls at least like v^-1 there (wings
// and the flanks of the core) it passes t_in at 2e-4 of v inside, which one evaluation confirms;
// only lines whose peak is just above the cut take a search of their own.
__device__ void cut_speeds(float a, float r, float* v_out, float* v_in) {
    const float t_out = r * (1.f - 1e-4f), t_in = r * (1.f + 1e-4f);
    float ge, lt;
    crossing(a, t_out, v_bound(a, t_out), &ge, &lt);
    *v_out = lt;
    const float vi = ge * (1.f - 2e-4f);
    if (ge > 0.f && voigt_H(vi, a) >= t_in) {
        *v_in = vi;
        return;
    }
    if (voigt_H(0.f, a) < t_in) {
        *v_in = -1.f;
        return;
    }
    crossing(a, t_in, v_bound(a, t_in), &ge, &lt);
    *v_in = ge < 0.f ? 0.f : ge;
}

// grid offsets d >= 0 at which |v| reaches vv, red side (d > 0: |v| = kv (1 - e^{-d lnq}))
// and blue side (|v| = kv (e^{d lnq} - 1)).
__device__ __forceinline__ float d_red(float vv, float kv, float lnq) {
    const float t = vv / kv;
    return t >= 1.f ? 1.0e9f : fminf(-log1pf(-t) / lnq, 1.0e9f);
}
__device__ __forceinline__ float d_blue(float vv, float kv, float lnq) { return fminf(log1pf(vv / kv) / lnq, 1.0e9f); }

constexpr unsigned char kDropped = 255;

// The tile kernel's constants of one kept (row, line), stored in bucket order so that a
// tile's candidates are one contiguous run of records (two 16-byte loads per line) instead of
// gathers from nine line-indexed arrays.  The inner cut window [ilo, ihi] is kept as its
// distances from the ends of the outer one, 16 bits each (the windows differ by about 2e-4 of
// their width); a line without an inner window, or with one further in than that, has none.
struct __align__(16) LineRec {
    int c;
    float f, kv, a;
    float srel;
    int jlo, jhi;
    unsigned in;
};
constexpr unsigned kNoInner = 0xffffffffu;
__device__ __forceinline__ unsigned pack_inner(int jlo, int jhi, int ilo, int ihi) {
    const int l = ilo - jlo, h = jhi - ihi;
    return ilo <= ihi && l < 65535 && h < 65535 ? (unsigned)l | ((unsigned)h << 16) : kNoInner;
}
// every point of [j0, j1] is inside the inner window
__device__ __forceinline__ bool inner_covers(int jlo, int jhi, unsigned in, int j0, int j1) {
    return in != kNoInner && jlo + (int)(in & 0xffffu) <= j0 && jhi - (int)(in >> 16) >= j1;
}

// Lists of the lines that k_prep lets through, per row (compact: every array is indexed by the
// position in the list).  The lines of a prep block are one run of the list, in line order.
struct PrepOut {
    int* surv;            // [n_sel][L] line indices
    int* nsurv;           // [n_sel] their number
    int2* run;            // [n_sel][nb] each prep block's run: first position, length
    float* srel;          // [n_sel][L]
    int4* win;            // [n_sel][L] jlo, jhi, ilo, ihi
    unsigned char* cls;   // [n_sel][L] width class, kDropped if the window misses the grid
    int* blkcnt;          // [n_sel][kNumClasses][nb]
};

// k_prep: one CTA of kPrepThreads threads per block of kPrepLines lines of one row.  Every line
// is tested: its peak against the cut threshold, then whether its wing can reach the grid.  With
// H <= 4a/(sqrt(pi) v^2) + exp(-v^2/4) (the convolution split at |t| = v/2) and 1/r = s_rel =
// e^rel, rel = ln S - ln t_p <= 88, a line stays below the cut beyond max(w, 2 sqrt(ln 2 + rel)),
// w^2 = 8 a s_rel/sqrt(pi), the second of which is below 19: a line whose nearest grid point
// lies at |v| = kv dist is dropped if that is above 22 and 3 per cent above w (k_windows drops
// exactly what is left).  The squares are compared, so the test costs one exponential and no
// logarithm, root or division: 3.4 -> 1.4 ms for 4e8 (row, line) pairs, and 0.94 ms for their bounds, of which
// it reads 8 B each (4 more of the few lines that can reach).  The lines that
// remain are appended, as one run per block in line order, to the row's list, and flagged for
// k_place.  The block's class counts, which k_windows adds to, start at zero here.
// BOUNDS: lnk0 holds upper bounds of ln kappa0 and lnS of ln(a S) (k_bounds; av is not read); lines that the
// full terms drop may be listed, k_windows drops them.
template <bool BOUNDS>
__global__ void __launch_bounds__(kPrepThreads) k_prep(int64_t L, size_t ld, RowGrids grids,
                                                       const int* __restrict__ species,
                                                       const float* __restrict__ dist, unsigned char* __restrict__ flag,
                                                       int n_sp, const SpConst* __restrict__ sc,
                                                       const float* __restrict__ lnS, const float* __restrict__ av,
                                                       const float* __restrict__ lnk0, const float* __restrict__ ln_tp,
                                                       int nb, PrepOut o) {
    static_assert(kPrepLines == 4 * kPrepThreads, "four lines per thread");
    constexpr int kWarps = kPrepThreads / 32;
    __shared__ int s_cnt[2][kWarps], s_base;
    const int s = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const size_t gL = grids.of(s).index * ld;
    const float ltp = ln_tp[s];
    // a block's four lines of the thread (rows are padded to a multiple of four); its bounds of ln kappa0
    // are read for the lines that pass the other test only
    struct Four {
        float4 k, s, a, d;
    };
    auto load = [&](int blk) {
        Four f{};
        const int64_t i0 = (int64_t)blk * kPrepLines + 4 * tid;
        if (blk < nb && i0 < L) {
            if (!BOUNDS) {
                f.k = __ldcs(reinterpret_cast<const float4*>(lnk0 + s * ld + i0));
                f.a = __ldg(reinterpret_cast<const float4*>(av + s * ld + i0));
            }
            f.s = __ldg(reinterpret_cast<const float4*>(lnS + s * ld + i0));
            f.d = __ldg(reinterpret_cast<const float4*>(dist + gL + i0));
        }
        return f;
    };
    Four next = load(blockIdx.x);
    float kv_min = INFINITY;   // of the row's species
    for (int p = lane; p < n_sp; p += 32) kv_min = fminf(kv_min, sc[(size_t)s * n_sp + p].kv);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) kv_min = fminf(kv_min, __shfl_xor_sync(0xffffffffu, kv_min, d));
    int par = 0;
    for (int blk = blockIdx.x; blk < nb; blk += gridDim.x, par ^= 1) {
        const Four f = next;
        next = load(blk + gridDim.x);
        const int64_t i0 = (int64_t)blk * kPrepLines + 4 * tid;
        if (tid < kNumClasses) o.blkcnt[((size_t)s * kNumClasses + tid) * nb + blk] = 0;
        const float lk[4] = {f.k.x, f.k.y, f.k.z, f.k.w}, ls[4] = {f.s.x, f.s.y, f.s.z, f.s.w};
        const float la[4] = {f.a.x, f.a.y, f.a.z, f.a.w}, di[4] = {f.d.x, f.d.y, f.d.z, f.d.w};
        // Peak and reach, the reach with the slowest species first; the few lines left take their own (off
        // the grid only) and, with bounds, their peak.  Each gather is issued for the four lines at
        // once: one after the other, inside the tests, they cost a block eight memory latencies.
        // (With bounds nothing is capped and a NaN keeps the line.)
        float w2[4], x[4];
        int sp[4];
        bool in[4];
        auto reaches = [&](float w, float need) { return need <= 22.f || (BOUNDS ? !(w < need * need) : w >= need * need); };
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            w2[k] = BOUNDS ? 8.f * kInvSqrtPi * 1.06f * __expf(ls[k] - ltp)
                           : 8.f * kInvSqrtPi * 1.06f * la[k] * __expf(fminf(ls[k] - ltp, 88.f));
            in[k] = i0 + k < L && (BOUNDS || lk[k] >= ltp) && reaches(w2[k], kv_min * di[k]);
        }
        unsigned reach = 0u;   // bit k: line i0 + k is kept
        bool more = false;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            reach |= in[k] ? 1u << k : 0u;
            more = more || (in[k] && (BOUNDS || di[k] > 0.f));
        }
        if (more) {
            reach = 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                sp[k] = in[k] ? __ldg(species + i0 + k) : 0;
                if (BOUNDS) x[k] = in[k] ? __ldg(lnk0 + s * ld + i0 + k) : 0.f;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float need = __ldg(&sc[(size_t)s * n_sp + sp[k]].kv) * di[k];
                if (in[k] && (di[k] <= 0.f || reaches(w2[k], need)) && (!BOUNDS || !(x[k] < ltp))) reach |= 1u << k;
            }
        }
        // the lines' places in the run: within the warp, then over the warps
        const int cnt = __popc(reach);
        int incl = cnt;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += y;
        }
        if (lane == 31) s_cnt[par][warp] = incl;
        __syncthreads();
        int before = 0, n = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const int c = s_cnt[par][w];
            if (w < warp) before += c;
            n += c;
        }
        if (n == 0) {
            if (tid == 0) o.run[(size_t)s * nb + blk] = make_int2(0, 0);
            continue;
        }
        if (tid == 0) {
            const int base = atomicAdd(&o.nsurv[s], n);
            s_base = base;
            o.run[(size_t)s * nb + blk] = make_int2(base, n);
        }
        __syncthreads();
        int pos = s_base + before + incl - cnt;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if ((reach >> k) & 1u) {
                o.surv[s * ld + pos++] = (int)(i0 + k);
                flag[gL + i0 + k] = 1;
            }
    }
}

// k_windows: the outer and inner cut windows of every listed line (crossing searches on the
// FP32 H), its width class.  Threads run over the row's list, so warps are dense whatever
// fraction of the lines the cheap bound kept.  A CTA first sorts its 256 lines by the tier of H
// at their expected crossing (far wing, continued fraction, core): a warp whose lanes need
// different tiers runs all of them at every evaluation.  The per-block class counts are integer
// atomics, combined first across the lanes of a warp that hold lines of the same prep block.
// BOUNDS: the list was made from bounds (k_prep): the lines take their full terms here, those whose
// peak is below the cut are dropped, and ln S and a are stored.
template <bool BOUNDS>
__global__ void __launch_bounds__(kPrepThreads, 3) k_windows(size_t ld, RowGrids grids, LineList lines,
                                                          const int* __restrict__ cpos, const float* __restrict__ fpos,
                                                          int n_sp, const RowConst* __restrict__ rc,
                                                          const SpConst* __restrict__ sc, float* lnS, float* av,
                                                          const float* __restrict__ ln_tp, int nb, PrepOut o) {
    constexpr int kWarps = kPrepThreads / 32;
    __shared__ unsigned char perm[kPrepThreads];
    __shared__ int cnt[4][kWarps];
    const int* __restrict__ species = lines.species;
    const int s = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = o.nsurv[s];
    const GridDesc gd = grids.of(s);
    const int N = gd.N;
    const float lnq = gd.lnq;
    const size_t gL = gd.index * ld;
    const float ltp = ln_tp[s];
    for (int base = blockIdx.x * kPrepThreads; base < n; base += gridDim.x * kPrepThreads) {
        {   // ---- sort by tier
            int cat = 3;
            if (base + tid < n) {
                const int64_t i = o.surv[s * ld + base + tid];
                const size_t q = s * ld + i;
                float ls, a;
                bool kept = true;
                if (BOUNDS) {
                    kept = line_terms(line_const(lines, i), rc[s], sc[(size_t)s * n_sp + species[i]], &ls, &a) >= ltp;
                    lnS[q] = ls;
                    av[q] = a;
                } else {
                    ls = __ldg(lnS + q);
                    a = __ldg(av + q);
                }
                const float rel = fminf(ls - ltp, 88.f);
                const float z2 = fmaxf(a * kInvSqrtPi * __expf(rel), rel) + a * a;
                cat = z2 >= 1600.f ? 0 : (z2 >= 36.f ? 1 : 2);
                if (!kept) {   // sorted behind the others
                    cat = 3;
                    o.cls[s * ld + base + tid] = kDropped;
                }
            }
            unsigned mine = 0u;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const unsigned m = __ballot_sync(0xffffffffu, cat == q);
                if (cat == q) mine = m;
                if (lane == 0) cnt[q][warp] = __popc(m);
            }
            __syncthreads();
            int off = __popc(mine & ((1u << lane) - 1u));
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int w = 0; w < kWarps; ++w)
                    if (q < cat || (q == cat && w < warp)) off += cnt[q][w];
            perm[off] = (unsigned char)tid;
            __syncthreads();
        }
        const int t = base + perm[tid];
        int live = 0;   // lines of the categories 0 to 2
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
            for (int w = 0; w < kWarps; ++w) live += cnt[q][w];
        int blk = 0, key2 = -1;
        if (tid < live) {
            const int64_t i = o.surv[s * ld + t];
            const size_t q = s * ld + i;
            blk = (int)(i / kPrepLines);
            const float rel = fminf((BOUNDS ? lnS[q] : __ldg(lnS + q)) - ltp, 88.f);
            const float r = expf(-rel);
            const int c = cpos[gL + i];
            const float f = fpos[gL + i], a = BOUNDS ? av[q] : __ldg(av + q), kv = sc[(size_t)s * n_sp + species[i]].kv;
            unsigned char cl = kDropped;
            const float srel = expf(rel);
            float vo, vi;
            cut_speeds(a, r, &vo, &vi);
            const float vo2 = vo * (1.f + 1e-5f);
            long long hi = (long long)c + (long long)floorf(fminf(f + d_red(vo2, kv, lnq), 1.0e9f)) + 2;
            long long lo = (long long)c + (long long)ceilf(fmaxf(f - d_blue(vo2, kv, lnq), -1.0e9f)) - 2;
            hi = hi > N - 1 ? N - 1 : hi;
            lo = lo < 0 ? 0 : lo;
            if (lo <= hi) {
                const int jlo = (int)lo, jhi = (int)hi;
                int ilo = 1, ihi = 0;
                // (s_rel a beyond FP32, s_rel near e^88 and a > 2: no inner window, so that no level interpolates the
                // line; its points multiply s_rel by H)
                if (vi >= 0.f && srel * a < INFINITY) {
                    const float vi2 = vi * (1.f - 1e-5f);
                    long long ih = (long long)c + (long long)floorf(fminf(f + d_red(vi2, kv, lnq), 1.0e9f)) - 2;
                    long long il = (long long)c + (long long)ceilf(fmaxf(f - d_blue(vi2, kv, lnq), -1.0e9f)) + 2;
                    ih = ih > jhi ? jhi : ih;
                    il = il < jlo ? jlo : il;
                    if (il <= ih) {
                        ilo = (int)il;
                        ihi = (int)ih;
                    }
                }
                const int key = c < -1 ? -1 : (c > N ? N : c);
                const int hw = max(jhi - key, key - jlo);
                cl = (unsigned char)(32 - __clz(hw));
                key2 = blk * kNumClasses + cl;
                o.srel[s * ld + t] = srel;
                o.win[s * ld + t] = make_int4(jlo, jhi, ilo, ihi);
            }
            o.cls[s * ld + t] = cl;
        }
        // kept lines per (prep block, class)
        const unsigned same = __match_any_sync(0xffffffffu, key2);
        if (key2 >= 0 && lane == __ffs(same) - 1)
            atomicAdd(&o.blkcnt[((size_t)s * kNumClasses + key2 % kNumClasses) * nb + blk], __popc(same));
        __syncthreads();   // perm and cnt are free for the next lines
    }
}

// k_scan_class: per (class, row), exclusive scan in place of the per-block counts of the
// class (one CTA each) and the class total; the row's number of profile evaluations starts at zero.
__global__ void __launch_bounds__(1024) k_scan_class(int nb, int* __restrict__ blkcnt, int* __restrict__ classcnt,
                                                     RowOut out) {
    __shared__ int wsum[32];
    __shared__ int carry;
    const int b = blockIdx.x, s = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int* row = blkcnt + ((size_t)s * kNumClasses + b) * nb;
    if (tid == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < nb; base += blockDim.x) {
        const int k = base + tid;
        const int v = k < nb ? row[k] : 0;
        int incl = v;
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += y;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const int t = lane < (int)(blockDim.x >> 5) ? wsum[lane] : 0;
            int ti = t;
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, ti, d);
                if (lane >= d) ti += y;
            }
            wsum[lane] = ti - t;
        }
        __syncthreads();
        const int c0 = carry;
        const int ex = c0 + wsum[warp] + incl - v;
        if (k < nb) row[k] = ex;
        __syncthreads();
        if (tid == (int)blockDim.x - 1) carry = ex + v;
        __syncthreads();
    }
    if (tid == 0) {
        classcnt[s * kNumClasses + b] = carry;
        unsigned long long* const ev = b == 0 ? out.ev_of(s) : nullptr;
        if (ev) *ev = 0;
    }
}

// lines of a row's classes before class b
__device__ __forceinline__ int class_base(const int* __restrict__ cnt, int b) {
    int acc = 0;
#pragma unroll
    for (int q = 0; q < kNumClasses - 1; ++q) acc += q < b ? cnt[q] : 0;
    return acc;
}

// k_scatter: stable placement of the kept lines into class buckets (centre order preserved): W
// warps per prep block's run of the row's list (one, or eight where the call has too few blocks to
// fill the GPU with one each), each taking a part of the run, 32 lines at a time; the lanes of
// one class rank themselves, and a warp keeps how many of each class are placed.  Blocks
// without kept lines cost one load.  The window lengths are added to the row's evaluations.
template <int W>
__global__ void __launch_bounds__(kPrepThreads) k_scatter(size_t ld, RowGrids grids, const int* __restrict__ species,
                                                          const int* __restrict__ cpos, const float* __restrict__ fpos,
                                                          int n_sp, const SpConst* __restrict__ sc,
                                                          const float* __restrict__ av, const int* __restrict__ blkoff,
                                                          const int* __restrict__ classcnt, int nb, const PrepOut o,
                                                          LineRec* __restrict__ rec, int* __restrict__ line,
                                                          RowOut out) {
    constexpr int kWarps = kPrepThreads / 32;
    static_assert(W == 1 || W == kWarps, "a run is one warp's or one CTA's");
    __shared__ int placed[kWarps][32];
    const int s = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int blk = blockIdx.x * (kWarps / W) + warp / W, part = warp % W;
    const int2 run = blk < nb ? o.run[(size_t)s * nb + blk] : make_int2(0, 0);
    if (run.y == 0) return;   // all of the run's warps
    const size_t sL = s * ld, gL = grids.of(s).index * ld;
    const int len = W == 1 ? run.y : 32 * ((run.y + 32 * W - 1) / (32 * W));   // lines of one warp
    const int t1 = min(run.x + run.y, run.x + (part + 1) * len), tb = run.x + part * len;
    const unsigned lt = (1u << lane) - 1u;
    int first = lane < kNumClasses
                    ? class_base(classcnt + s * kNumClasses, lane) + blkoff[((size_t)s * kNumClasses + lane) * nb + blk]
                    : 0;
    if (W > 1) {   // the lines of each class in the parts before this one
        placed[warp][lane] = 0;
        __syncwarp();
        for (int t0 = tb; t0 < t1; t0 += 32) {
            const int b = t0 + lane < t1 ? (int)o.cls[sL + t0 + lane] : (int)kDropped;
            const unsigned same = __match_any_sync(0xffffffffu, b);
            if (b < kNumClasses && (same & lt) == 0u) placed[warp][b] += __popc(same);
            __syncwarp();
        }
        __syncthreads();
        for (int v = 0; v < part; ++v) first += placed[v][lane];
        __syncthreads();
    }
    placed[warp][lane] = first;
    __syncwarp();
    unsigned long long len_sum = 0;
    for (int t0 = tb; t0 < t1; t0 += 32) {
        const int t = t0 + lane;
        const int b = t < t1 ? (int)o.cls[sL + t] : (int)kDropped;
        const unsigned same = __match_any_sync(0xffffffffu, b);
        const int lrank = __popc(same & lt);
        if (b < kNumClasses) {
            const int i = o.surv[sL + t];
            const int4 w = o.win[sL + t];
            LineRec r;
            r.c = cpos[gL + i];
            r.f = fpos[gL + i];
            r.kv = sc[(size_t)s * n_sp + species[i]].kv;
            r.a = av[sL + i];
            r.srel = o.srel[sL + t];
            r.jlo = w.x;
            r.jhi = w.y;
            r.in = pack_inner(w.x, w.y, w.z, w.w);
            len_sum += (unsigned long long)(w.y - w.x + 1);
            rec[sL + placed[warp][b] + lrank] = r;
            line[sL + placed[warp][b] + lrank] = i;
        }
        __syncwarp();
        if (b < kNumClasses && lrank == 0) placed[warp][b] += __popc(same);
        __syncwarp();
    }
    unsigned long long* const ev = out.ev_of(s);
    if (ev) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) len_sum += __shfl_down_sync(0xffffffffu, len_sum, d);
        if (lane == 0 && len_sum) atomicAdd(ev, len_sum);
    }
}

// ---------------------------------------------------------------------------
// The profile kernel.  A tile of PTS * THREADS grid points is processed by one CTA:
// thread t owns the points J0 + k THREADS + t, k = 0..PTS-1.
struct RowDesc {
    int N, nT, tile;
    float lnq, q1, q2;          // expm1(-x)/(-x) ~ 1 + d (q1 + d q2), x = d lnq
    const float* ln_tp;         // ln of the cut threshold t_p (outputs are t_p * sum of s_rel H)
    int* cum;                   // [kNumClasses][nT + 3]
    const LineRec* rec;         // [L] the bucketed lines
    const int* line;            // [L] their indices in the list
    float* out;                 // [N]
};

// k_ranges: cum[b][ts] of a row = position of its first line of class b whose centre key (its grid
// index, off-grid centres clamped to -1 and N) is >= (ts - 1) * tile, ts = 0 .. nT + 2.  rows: a
// descriptor per row, or null: `one` for all, with their arrays following one another.
__global__ void k_ranges(int n_sel, size_t ld, RowDesc one, const RowDesc* __restrict__ rows,
                         const int* __restrict__ classcnt) {
    const int s = blockIdx.y;
    RowDesc g = one;
    if (rows) {
        g = rows[s];
    } else {
        g.cum += (size_t)s * kNumClasses * (g.nT + 3);
        g.rec += s * ld;
    }
    const int t = blockIdx.x * blockDim.x + threadIdx.x, W = g.nT + 3;
    if (t >= kNumClasses * W) return;
    const int b = t / W, ts = t - b * W;
    const int base = class_base(classcnt + s * kNumClasses, b), n = classcnt[s * kNumClasses + b];
    const LineRec* k = g.rec + base;
    const long long thr = (long long)(ts - 1) * g.tile;
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (min(max(k[mid].c, -1), g.N) < thr) lo = mid + 1; else hi = mid;
    }
    g.cum[t] = base + lo;
}

// ---------------------------------------------------------------------------
// Wing sums by interpolation.
//
// Seen from a stretch of the grid that lies at least its own length away from the line's
// centre, a profile is smooth: s_rel H has its nearest singularity (the centre) at three
// half-lengths from the stretch's middle, so its Chebyshev interpolant converges like
// 5.8^-n.  With kNodes = 12 nodes the interpolant of 1/v^2 is within 2.3e-8 of it anywhere on
// the stretch (10 nodes: 6.7e-7, 8: 1.8e-5), below the 1e-6 of the profile formulas.  That is
// so while v is linear in the grid index.  Blueward of a centre v grows like e^x, x = ln lambda, and a
// stretch that is long in x takes more nodes: 2.1e-7 where it spans 1 in x, 7.9e-7 at 1.5, 3.3e-6 at 2,
// 3.5e-4 at 3.5 (the interpolant restated in FP64, the centre one span beyond the end).  So a
// stretch of more than kMaxStretch is not interpolated: tiles of 2048 points below R = 2048, of 4096
// below 4096, warp parts below an eighth of that.  The sum
// over such lines is therefore formed at the nodes only, and interpolated once per tile:
// 12 evaluations per (line, stretch) instead of one per point.
//
// Two stretches are used, the CTA's tile (level 0) and a warp's part of it (level 1).  Lines
// that neither level takes (centre too close, window edge inside, too small |z|) are
// evaluated point by point.
constexpr int kNodes = 12;
constexpr float kMaxStretch = 1.f;   // in ln lambda
// cos(i pi / 24): node k of a stretch is at (1 + x_k)/2 of its length, x_k = cos((2k + 1) pi / 24),
// and T_m(x_k) = cos(m (2k + 1) pi / 24)
__constant__ float c_cos24[48] = {
    1.f, 0.991444886f, 0.965925813f, 0.923879504f, 0.866025388f, 0.793353319f, 0.707106769f, 0.60876143f,
    0.5f, 0.382683426f, 0.258819044f, 0.130526185f, 0.f, -0.130526185f, -0.258819044f, -0.382683426f,
    -0.5f, -0.60876143f, -0.707106769f, -0.793353319f, -0.866025388f, -0.923879504f, -0.965925813f, -0.991444886f,
    -1.f, -0.991444886f, -0.965925813f, -0.923879504f, -0.866025388f, -0.793353319f, -0.707106769f, -0.60876143f,
    -0.5f, -0.382683426f, -0.258819044f, -0.130526185f, 0.f, 0.130526185f, 0.258819044f, 0.382683426f,
    0.5f, 0.60876143f, 0.707106769f, 0.793353319f, 0.866025388f, 0.923879504f, 0.965925813f, 0.991444886f};
// and what FP32 rounds off
__constant__ float c_cos24_lo[48] = {
    0.f, -2.43569325e-08f, 1.35678162e-08f, 2.83074897e-08f, 1.55436251e-08f, 2.11231441e-08f, 1.21016175e-08f, -7.77961473e-10f,
    0.f, 6.22335072e-09f, 1.46619872e-09f, 7.18434601e-09f, 0.f, -7.18434601e-09f, -1.46619872e-09f, -6.22335072e-09f,
    0.f, 7.77961473e-10f, -1.21016175e-08f, -2.11231441e-08f, -1.55436251e-08f, -2.83074897e-08f, -1.35678162e-08f, 2.43569325e-08f,
    0.f, 2.43569325e-08f, -1.35678162e-08f, -2.83074897e-08f, -1.55436251e-08f, -2.11231441e-08f, -1.21016175e-08f, 7.77961473e-10f,
    0.f, -6.22335072e-09f, -1.46619872e-09f, -7.18434601e-09f, 0.f, 7.18434601e-09f, 1.46619872e-09f, 6.22335072e-09f,
    0.f, -7.77961473e-10f, 1.21016175e-08f, 2.11231441e-08f, 1.55436251e-08f, 2.83074897e-08f, 1.35678162e-08f, -2.43569325e-08f};

// The offset v of a line at the points of a stretch starting D points from its centre:
// v = G (kv B) + kv E1 with E1 = expm1(-D ln q), B = 1 + E1 and G = expm1(-delta ln q) for the
// point delta points into the stretch (the exact split of expm1).  Both terms are at most
// the larger of the stretch's span and the centre's distance, so with the centre at least the
// span away v keeps about 2e-7 relative accuracy.
struct Wing {
    float kvE, kvB;      // kv E1, kv B
    float dist;          // distance [points] of the centre from the stretch, < 0 inside
    float zmin2, zmax2;  // smallest and largest |z|^2 on the stretch
};
// expm1(x): its series to x^6 for |x| <= 1/8 (below 8e-10 of it; stretches within a ninth of the wavelength of
// the centre, which almost all are), a quarter of expm1f's instructions
__device__ __forceinline__ float expm1_near(float x) {
    if (fabsf(x) <= 0.125f)
        return x * fmaf(x, fmaf(x, fmaf(x, fmaf(x, fmaf(x, 1.f / 720.f, 1.f / 120.f), 1.f / 24.f), 1.f / 6.f), 0.5f), 1.f);
    return expm1f(x);
}
// span = its number of points - 1, gend = G at its end
__device__ __forceinline__ Wing wing(int J, int c, float f, float kv, float A, float lnq, float span, float gend) {
    Wing w;
    const float D = (float)(J - c) - f;
    const float E1 = expm1_near(-D * lnq);
    w.kvE = kv * E1;
    w.kvB = kv + w.kvE;
    const float v0 = fabsf(w.kvE), v1 = fabsf(fmaf(gend, w.kvB, w.kvE));
    w.dist = fmaxf(D, -(D + span));
    const float vm = fminf(v0, v1), vx = fmaxf(v0, v1);
    w.zmin2 = fmaf(vm, vm, A);
    w.zmax2 = fmaf(vx, vx, A);
    return w;
}
// The rational far form s_rel H = sk / (|z|^2 - 3/2), sk = s_rel a / sqrt(pi): its relative error is
// below (2 + 2 a^2)/|z|^4 (the asymptotic series of H to order |z|^-4), so it is used where
// that is at most 1e-6 on the whole stretch; |z|^2 <= 1e18 keeps the product of two denominators
// finite.
__device__ __forceinline__ bool rational_ok(const Wing& w, float A) {
    return w.zmin2 * w.zmin2 >= 1.0e6f * fmaf(2.f, A, 2.f) && w.zmax2 <= 1.0e18f;
}
// acc[k] += s_rel H at the nodes (G[k]: expm1(-delta_k ln q)), rational form, two nodes per
// reciprocal in packed FP32: r = 1/(D_0 D_1), sk/D_0 = sk r D_1, sk/D_1 = sk r D_0, the pair's sums
// held as {acc_{2j+1}, acc_{2j}}.  Per pair three packed FFMAs, two FMULs and one reciprocal.
__device__ __forceinline__ void nodes_rational(const Wing& w, float A, float sk, const float* G, float2 (&acc)[kNodes / 2]) {
    const float2 B2 = dup2(w.kvB), E2 = dup2(w.kvE), C2 = dup2(A - 1.5f);
#pragma unroll
    for (int j = 0; j < kNodes / 2; ++j) {
        const float2 v = ffma2(make_float2(G[2 * j], G[2 * j + 1]), B2, E2);
        const float2 D = ffma2(v, v, C2);
        const float sr = sk * rcp_approx(D.x * D.y);
        acc[j] = ffma2(dup2(sr), D, acc[j]);
    }
}
// the same by the series (LOW: a^2 <= 2)
template <bool LOW>
__device__ __forceinline__ void nodes_series(const Wing& w, float A, float sk, const float* G, float2 (&acc)[kNodes / 2]) {
    const float2 B2 = dup2(w.kvB), E2 = dup2(w.kvE), A2 = dup2(A), S2 = dup2(sk), zero = dup2(0.f);
    const float2 k2 = dup2(series_k2(A)), k3 = dup2(series_k3(A)), k4 = dup2(series_k4(A));
#pragma unroll
    for (int j = 0; j < kNodes / 2; ++j) {
        const float2 v = ffma2(make_float2(G[2 * j], G[2 * j + 1]), B2, E2);
        const float2 Z = ffma2(v, v, A2);
        const float r = rcp_approx(Z.x * Z.y);
        const float2 t = make_float2(r * Z.x, r * Z.y);   // {1/Z_{2j+1}, 1/Z_{2j}}
        float2 h;
        if (LOW) {
            h = ffma2(t, ffma2(t, ffma2(t, k4, k3), k2), dup2(1.5f));
        } else {
            const float2 s = ffma2(A2, t, zero);
            const float2 c1 = ffma2(s, dup2(-2.f), dup2(1.5f));
            const float2 c2 = ffma2(s, ffma2(s, dup2(12.f), dup2(-15.f)), dup2(3.75f));
            const float2 c3 = ffma2(s, ffma2(s, ffma2(s, dup2(-120.f), dup2(210.f)), dup2(-105.f)), dup2(13.125f));
            h = ffma2(t, ffma2(t, c3, c2), c1);
        }
        h = ffma2(t, h, dup2(1.f));
        acc[j] = ffma2(ffma2(t, S2, zero), h, acc[j]);
    }
}

// sum of one value over the warp, in every lane
__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    return v;
}

// total += y: Kahan-compensated, or a plain sum for the naive variant
template <int PREC>
__device__ __forceinline__ void fold(float& sum, float& comp, float v) {
    if (PREC == MPSA_PREC_FP32_COMPENSATED) {
        const float y = v - comp;
        const float t = sum + y;
        comp = (t - sum) - y;
        sum = t;
    } else {
        sum += v;
    }
}

// Add a warp's node sums (over its lanes) to the warp's totals F[k] = {sum, comp}; clears acc.
template <int PREC>
__device__ __forceinline__ void fold_nodes(float2 (&acc)[kNodes / 2], float2* F, int lane) {
    float mine = 0.f;
#pragma unroll
    for (int j = 0; j < kNodes / 2; ++j) {
        const float hi = warp_sum_f(acc[j].x), lo = warp_sum_f(acc[j].y);   // nodes 2j + 1 and 2j
        if (lane == 2 * j) mine = lo;
        if (lane == 2 * j + 1) mine = hi;
        acc[j] = make_float2(0.f, 0.f);
    }
    if (lane < kNodes) {
        float2 q = F[lane];
        fold<PREC>(q.x, q.y, mine);
        F[lane] = q;
    }
}

// {hi, lo} += v (lo takes the rounding error of hi + v; Knuth's two-sum)
__device__ __forceinline__ void acc_pair(float& hi, float& lo, float v) {
    const float t = __fadd_rn(hi, v), z = __fsub_rn(t, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, z)), __fsub_rn(v, z)));
    hi = t;
}

// Chebyshev coefficients c_m = (2 - [m = 0])/n sum_k F_k T_m(x_k) of the node totals F_k = fx - fy,
// node k in lane k of the warp; lane m < n gets c_m.  In FP32 pairs (products and sums with their
// errors): FP64 has 1/64 of the FP32 rate here, and with it the two transforms cost a tile some 5 us.
__device__ __forceinline__ float cheb_coefs(float fx, float fy, int lane) {
    float hi = 0.f, lo = 0.f;
#pragma unroll
    for (int k = 0; k < kNodes; ++k) {
        const float x = __shfl_sync(0xffffffffu, fx, k), y = __shfl_sync(0xffffffffu, fy, k);
        const int i = (lane * (2 * k + 1)) % 48;
        const float t = c_cos24[i], tl = c_cos24_lo[i], pr = __fmul_rn(t, x);
        acc_pair(hi, lo, pr);
        lo += fmaf(t, x, -pr) + fmaf(tl, x, -t * y);
    }
    return (hi + lo) * ((lane == 0 ? 1.f : 2.f) / kNodes);
}

// Clenshaw sum of the Chebyshev series c[0..kNodes) at x
__device__ __forceinline__ float clenshaw(const float* c, float x) {
    float b1 = 0.f, b2 = 0.f;
    const float x2 = 2.f * x;
#pragma unroll
    for (int m = kNodes - 1; m >= 1; --m) {
        const float b = fmaf(x2, b1, c[m] - b2);
        b2 = b1;
        b1 = b;
    }
    return fmaf(x, b1, c[0] - b2);
}

// A line that a warp evaluates point by point on its part of the tile: window edges inside the
// part, centres on or next to it.  Window [lo, hi] relative to Js, kind one of
//   kPtRat     rational form on the whole part, v from the expm1 split (u.z = kv E1, u.w = kv B)
//   kPtWing    the series of H on the whole part, v from the expm1 split, a^2 <= 2
//   kPtNear    centre within the part's length: v = kv (x - x^2/2 + x^3/6)-like series (|x| <= 0.01, the
//              rest is below 5e-8 of it); the pairs of points jc0..jc1 (|z|^2 < 64, in u.z and u.w
//              as integers) by voigt_small2 or, for a > 0.03, the Gauss-Hermite tiers; the others
//              by the series of H (grids of at most 2 in v per point, so that no point of
//              those pairs is beyond |v| = 10)
//   kPtGen     any other case, decided point by point
// with kPtChk where the part is not inside the inner window: a point then takes the line iff
// s_rel H >= 1.
struct __align__(16) PointRec {
    float ci, f, klnq, A;          // ci = c - Js (exact)
    float sk, srel, kvE, kvB;
    int lo, hi, kind;
    float a;
};
constexpr int kPtRat = 0, kPtWing = 1, kPtNear = 2, kPtGen = 3, kPtKind = 3, kPtAway = 4, kPtChk = 8;
constexpr int kPtRecs = 32;    // records a warp holds

// two neighbouring points: x[2p], x[2p + 1] += l where l passes the cut
__device__ __forceinline__ void add_pair(float2* x, int p, float2 l, float floor1) {
    l.x = l.x >= floor1 ? l.x : 0.f;
    l.y = l.y >= floor1 ? l.y : 0.f;
    x[p] = fadd2(x[p], l);
}
// offsets d = j - c - f of the points j = 2p, 2p + 1
__device__ __forceinline__ float2 pair_offsets(int p, const float4 q) {
    const float j = (float)(2 * p);
    return fadd2(fadd2(make_float2(j, j + 1.f), dup2(-q.x)), dup2(-q.y));
}
__device__ __forceinline__ float2 pair_v(float2 d, const float4 q, float q1, float q2) {
    return fmul2(dup2(q.z), fmul2(d, ffma2(d, ffma2(d, dup2(q2), dup2(q1)), dup2(1.f))));
}
// sk times the series of H at two points (a^2 <= 2), one reciprocal for both
__device__ __forceinline__ float2 pair_series(float2 v, float A, float sk, float k2, float k3, float k4) {
    const float2 Z = ffma2(v, v, dup2(A));
    const float r = rcp_approx(Z.x * Z.y);
    const float2 y = make_float2(r * Z.y, r * Z.x);
    const float2 h = ffma2(y, ffma2(y, ffma2(y, ffma2(y, dup2(k4), dup2(k3)), dup2(k2)), dup2(1.5f)), dup2(1.f));
    return fmul2(fmul2(dup2(sk), y), h);
}

// kPtNear's core, the pairs p0..p1, by voigt_small2 (TINY: a <= 3e-4)
template <bool TINY>
__device__ __forceinline__ void add_core(float2* x, int p0, int p1, int lane, const float4 p, float srel, float a,
                                         float floor1, float q1, float q2) {
#pragma unroll 1
    for (int i = p0 + lane; i <= p1; i += 32)
        add_pair(x, i, fmul2(dup2(srel), voigt_small2<TINY>(pair_v(pair_offsets(i, p), p, q1, q2), p.w, a)), floor1);
}

// One record added to the warp's points x[0..last].  A lane takes two neighbouring points at a
// time, in packed FP32, and the lanes 64 consecutive points of the window, so a narrow window
// costs no idle segments and no two lanes share a point.  (Points of a pair outside the window
// fail the test of the cut by its margin; points past the part's end are never stored.)  Every
// case has a loop of its own without branches: one loop deciding per point spent as many integer
// and control instructions as FP32 ones.  The kernel is bound by instruction issue; points one at
// a time took 16.5 ms for two table rows, pairs 14.3 ms.  Gp[j] = expm1(-j ln q).
__device__ __forceinline__ void add_points(const PointRec& r, float* xs, const float* Gs, int last, int lane, float q1,
                                           float q2, float lnq) {
    const int4 w = *reinterpret_cast<const int4*>(&r.lo);
    const float4 u = *reinterpret_cast<const float4*>(&r.sk);
    const float4 p = *reinterpret_cast<const float4*>(&r.ci);
    const float floor1 = (w.z & kPtChk) ? 1.f : 0.f;
    const int lo = max(w.x, 0), hi = min(w.y, last);
    const int kind = w.z & kPtKind;
    const float a = __int_as_float(w.w);
    float2* const x = reinterpret_cast<float2*>(xs);
    const float2* const Gp = reinterpret_cast<const float2*>(Gs);
    const int p0 = lo >> 1, p1 = hi >> 1;
    if (kind == kPtRat) {
        const float2 E = dup2(u.z), B = dup2(u.w), C = dup2(p.w - 1.5f);
#pragma unroll 1
        for (int i = p0 + lane; i <= p1; i += 32) {
            const float2 v = ffma2(Gp[i], B, E);
            const float2 D = ffma2(v, v, C);
            const float sr = u.x * rcp_approx(D.x * D.y);
            add_pair(x, i, make_float2(sr * D.y, sr * D.x), floor1);
        }
    } else if (kind == kPtNear) {
        const int c0 = max(p0, __float_as_int(u.z) >> 1), c1 = min(p1, __float_as_int(u.w) >> 1);
        // the pairs outside the core, left then right, as one sequence; no core: all of them
        const int nl = c0 <= c1 ? c0 - p0 : p1 - p0 + 1, gap = c0 <= c1 ? c1 - c0 + 1 : 0, n = p1 - p0 + 1 - gap;
        const float k2 = series_k2(p.w), k3 = series_k3(p.w), k4 = series_k4(p.w);
#pragma unroll 1
        for (int t = lane; t < n; t += 32) {
            const int i = p0 + t + (t >= nl ? gap : 0);
            add_pair(x, i, pair_series(pair_v(pair_offsets(i, p), p, q1, q2), p.w, u.x, k2, k3, k4), floor1);
        }
        if (a <= kTinyA) {
            add_core<true>(x, c0, c1, lane, p, u.y, a, floor1, q1, q2);
        } else if (a <= kSmallA) {
            add_core<false>(x, c0, c1, lane, p, u.y, a, floor1, q1, q2);
        } else {
#pragma unroll 1
            for (int i = c0 + lane; i <= c1; i += 32) {
                const float2 v = pair_v(pair_offsets(i, p), p, q1, q2);
                add_pair(x, i, make_float2(u.y * voigt_inner_tiers(v.x, a), u.y * voigt_inner_tiers(v.y, a)), floor1);
            }
        }
    } else if (kind == kPtWing) {
        const float k2 = series_k2(p.w), k3 = series_k3(p.w), k4 = series_k4(p.w);
        const float2 E = dup2(u.z), B = dup2(u.w);
#pragma unroll 1
        for (int i = p0 + lane; i <= p1; i += 32)
            add_pair(x, i, pair_series(ffma2(Gp[i], B, E), p.w, u.x, k2, k3, k4), floor1);
    } else {
#pragma unroll 1
        for (int j = lo + lane; j <= hi; j += 32) {
            float v;
            if (w.z & kPtAway) v = fmaf(Gs[j], u.w, u.z);
            else v = p.z / lnq * expm1f(-(((float)j - p.x) - p.y) * lnq);
            const float l = u.y * voigt_point(v, a);
            if (l >= floor1) xs[j] += l;
        }
    }
}

// One tile of one row.  Called by the grid kernel (one tile per CTA, or up to S CTAs per tile that
// take every S-th chunk of the tile's candidate lines, sp = 0..S-1, when a call has too few
// tiles to fill the GPU; *s_used says how many did) and by the persistent kernel (a loop over a work list).
//
// Candidate lines are taken THREADS at a time, one per thread: a thread adds its line to the
// node sums of the tile (level 0) in its own registers, so that a line costs its set-up and 12
// evaluations once, with no broadcast.  Lines that the tile cannot take are queued in shared
// memory (in candidate order); when the queue holds more than kQueue lines every warp runs
// over it, one line per lane, for its own part of the tile (level 1), and the lines that the
// part cannot take are gathered (kPtRecs a warp) and evaluated at its points by the whole warp.
//
// FP32 partial sums run over at most 64 lines (level 0, points) or 72 lines (level 1)
// and are folded into Kahan-compensated totals in shared memory.
constexpr int kSplitChunks = 64;   // chunks of candidates that are worth a CTA of their own
constexpr int kQueue = 2048;   // queued lines at which a tile turns to level 1

template <int PREC, int PTS, int THREADS>
__device__ __forceinline__ void tile_body(const RowDesc& g, int J0, int size, int sp = 0, int S = 1,
                                          int S_free = 1, int* s_used = nullptr) {
    constexpr int TILE = PTS * THREADS, WARPS = THREADS / 32, QCAP = THREADS + kQueue;
    __shared__ int sQ[QCAP];
    __shared__ PointRec sP[WARPS][kPtRecs];
    __shared__ __align__(8) float sX[WARPS][32 * PTS];   // sums of the gathered records at the warp's points
    __shared__ __align__(8) float sGp[32 * PTS];         // expm1(-j ln q) at the points j of a warp's part
    __shared__ float sG0[kNodes], sG1[WARPS][kNodes];
    __shared__ float2 sF0[WARPS][kNodes], sF1[WARPS][kNodes];   // node totals {sum, comp}
    __shared__ float sC0[kNodes], sC1[WARPS][kNodes];           // their Chebyshev coefficients
    __shared__ int sCnt[2][WARPS];
    __shared__ int sBeg[kNumClasses], sEnd[kNumClasses];        // each class's candidates
    __shared__ float sSum[PTS][THREADS];
    __shared__ float sComp[PREC == MPSA_PREC_FP32_COMPENSATED ? PTS : 1][THREADS];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const float lnq = g.lnq;
    // the tile's points on the grid, [J0, Te], and the warp's part of them, [Js, Je] (npt segments of
    // 32): a short tile is shared out over all warps
    const int Te = min(J0 + size, g.N) - 1;
    const int sub = 32 * ((Te - J0 + 32 * WARPS) / (32 * WARPS)), npt = sub / 32;
    const int Js = J0 + warp * sub, Je = min(Js + sub - 1, Te);
    const bool active = Js <= Te;
    const float span0 = (float)(Te - J0), span1 = active ? (float)(Je - Js) : 0.f;
    const float gend0 = expm1f(-span0 * lnq), gend1 = expm1f(-span1 * lnq);
    // a centre this far from the tile, or the part, is taken by interpolation
    const float far0 = span0 * lnq <= kMaxStretch ? span0 : INFINITY, far1 = span1 * lnq <= kMaxStretch ? span1 : INFINITY;
    if (lane < kNodes) {
        const float x = 0.5f + 0.5f * c_cos24[2 * lane + 1];
        sG1[warp][lane] = expm1f(-span1 * x * lnq);
        if (warp == 0) sG0[lane] = expm1f(-span0 * x * lnq);
        sF0[warp][lane] = sF1[warp][lane] = make_float2(0.f, 0.f);
    }
    if (tid < kNumClasses) {   // all classes at once: one memory latency instead of one per class
        const int reach = 1 << tid;
        const int tlo = max(floordiv(J0 - reach + 1, TILE), -1);
        const int thi = min(floordiv(Te + reach - 1, TILE), g.nT);
        const int* cum = g.cum + (size_t)tid * (g.nT + 3);
        sBeg[tid] = tlo <= thi ? cum[tlo + 1] : 0;
        sEnd[tid] = tlo <= thi ? cum[thi + 2] : 0;
    }
    for (int t = tid; t < 32 * PTS; t += THREADS) sGp[t] = expm1f(-(float)t * lnq);
#pragma unroll
    for (int k = 0; k < PTS; ++k) {
        sSum[k][tid] = 0.f;
        (&sX[0][0])[k * THREADS + tid] = 0.f;
        if (PREC == MPSA_PREC_FP32_COMPENSATED) sComp[k][tid] = 0.f;
    }
    __syncthreads();
    if (S > 1) {   // as many of the tile's CTAs as its candidates are worth
        int chunks = 0;
        for (int b = 0; b < kNumClasses; ++b) chunks += (sEnd[b] - sBeg[b] + THREADS - 1) / THREADS;
        S = max(1, max(min(S_free, chunks), min(S, chunks / kSplitChunks)));
        if (sp == 0 && tid == 0) *s_used = S;
        if (sp >= S) return;
    }

    // the warp's gathered point records at every segment of its part
    auto points = [&](int n) {
        __syncwarp();
        for (int i = 0; i < n; ++i) {
            add_points(sP[warp][i], sX[warp], sGp, Je - Js, lane, g.q1, g.q2, lnq);
            __syncwarp();
        }
        for (int k = 0; k < npt; ++k) {
            float dummy = 0.f;
            fold<PREC>(sSum[k][tid], PREC == MPSA_PREC_FP32_COMPENSATED ? sComp[k][tid] : dummy, sX[warp][32 * k + lane]);
            sX[warp][32 * k + lane] = 0.f;
        }
        __syncwarp();
    };
    // level 1 and the points, over the queued lines
    auto flush = [&](int n) {
        float2 acc[kNodes / 2];
#pragma unroll
        for (int j = 0; j < kNodes / 2; ++j) acc[j] = make_float2(0.f, 0.f);
        int np = 0;
        for (int i0 = 0; i0 < n; i0 += 32) {
            const int i = i0 + lane;
            bool direct = false, rat = false, ser = false;
            Wing w{};
            int4 r0, r1;
            float f = 0.f, kv = 0.f, a = 0.f, A = 0.f, sk = 0.f;
            bool inside = false;
            if (i < n) {
                const int4* rp = reinterpret_cast<const int4*>(g.rec + sQ[i]);
                r0 = __ldg(rp), r1 = __ldg(rp + 1);
                if (r1.z >= Js && r1.y <= Je) {
                    f = __int_as_float(r0.y), kv = __int_as_float(r0.z), a = __int_as_float(r0.w);
                    A = a * a;
                    sk = __int_as_float(r1.x) * a * kInvSqrtPi;
                    w = wing(Js, r0.x, f, kv, A, lnq, span1, gend1);
                    inside = inner_covers(r1.y, r1.z, (unsigned)r1.w, Js, Je);
                    const bool smooth = inside && w.dist > far1;
                    const bool ra = rational_ok(w, A);
                    rat = smooth && ra;
                    ser = smooth && !ra && w.zmin2 >= (A <= kSeriesA ? kSeriesZ2Low : kSeriesZ2) && w.zmax2 <= 1.0e18f;
                    direct = !rat && !ser;
                }
            }
            if (rat) nodes_rational(w, A, sk, sG1[warp], acc);
            if (__any_sync(0xffffffffu, ser)) {
                if (__all_sync(0xffffffffu, !ser || A <= kSeriesA)) {
                    if (ser) nodes_series<true>(w, A, sk, sG1[warp], acc);
                } else {
                    if (ser) nodes_series<false>(w, A, sk, sG1[warp], acc);
                }
            }
            const unsigned m = __ballot_sync(0xffffffffu, direct);
            if (np + __popc(m) > kPtRecs) {
                points(np);
                np = 0;
            }
            if (direct) {
                const bool away = w.dist > far1;
                PointRec p;
                p.ci = (float)(r0.x - Js);
                p.f = f;
                p.klnq = kv * lnq;
                p.A = A;
                p.sk = sk;
                p.srel = __int_as_float(r1.x);
                p.kvE = w.kvE;
                p.kvB = w.kvB;
                p.lo = r1.y - Js;
                p.hi = r1.z - Js;
                p.a = a;
                int kind = kPtGen;
                if (away && sk < INFINITY && rational_ok(w, A)) {   // (sk beyond FP32: a > 2, so the next two don't take it)
                    kind = kPtRat;
                } else if (A <= kSeriesA && away && w.zmin2 >= kSeriesZ2Low && w.zmax2 <= 1.0e18f) {
                    kind = kPtWing;
                } else if (A <= kSeriesA && !away && (span1 + fmaxf(w.dist, 0.f) + 1.f) * lnq <= 0.01f &&
                           w.zmax2 <= 1.0e18f && p.klnq <= 2.f) {
                    kind = kPtNear;
                    // |z| = 8 at this many points from the centre (v is linear to 0.5 per cent there)
                    const float h = fminf(sqrtf(kSeriesZ2Low - A) / p.klnq * 1.005f, 1.0e6f), x0 = p.ci + f;
                    p.kvE = __int_as_float((int)ceilf(x0 - h));
                    p.kvB = __int_as_float((int)floorf(x0 + h));
                }
                p.kind = kind | (away ? kPtAway : 0) | (inside ? 0 : kPtChk);
                sP[warp][np + __popc(m & ((1u << lane) - 1u))] = p;
            }
            np += __popc(m);
        }
        if (np > 0) points(np);
        fold_nodes<PREC>(acc, sF1[warp], lane);
    };

    float2 acc0[kNodes / 2];
#pragma unroll
    for (int j = 0; j < kNodes / 2; ++j) acc0[j] = make_float2(0.f, 0.f);
    int chunk = 0;    // running chunk index over the classes: this CTA takes chunk % S == sp
    int nq = 0;       // queued lines
    int par = 0, run = 0;
    int b = -1, base = 0, end = 0;   // class, next candidate, end of the class's candidates
    for (bool more = true; more;) {
        // ---- the next chunk of candidates (CTA-uniform)
        int pos0 = -1;
        while (pos0 < 0) {
            if (base < end) {
                if (chunk++ % S == sp) pos0 = base;
                base += THREADS;
            } else if (++b < kNumClasses) {
                base = sBeg[b];
                end = sEnd[b];
            } else {
                more = false;
                break;
            }
        }
        if (more) {
            // ---- level 0: one candidate line per thread
            const int pos = pos0 + tid;
            bool queue = false;
            if (pos < end) {
                const int4* rp = reinterpret_cast<const int4*>(g.rec + pos);
                const int4 r0 = __ldg(rp), r1 = __ldg(rp + 1);
                if (r1.z >= J0 && r1.y <= Te) {
                    const float a = __int_as_float(r0.w), A = a * a;
                    const Wing w = wing(J0, r0.x, __int_as_float(r0.y), __int_as_float(r0.z), A, lnq, span0, gend0);
                    if (inner_covers(r1.y, r1.z, (unsigned)r1.w, J0, Te) && w.dist > far0 && rational_ok(w, A))
                        nodes_rational(w, A, __int_as_float(r1.x) * a * kInvSqrtPi, sG0, acc0);
                    else
                        queue = true;
                }
            }
            // ---- queue the others, in candidate order
            const unsigned bm = __ballot_sync(0xffffffffu, queue);
            if (lane == 0) sCnt[par][warp] = __popc(bm);
            __syncthreads();
            const unsigned cnt = lane < WARPS ? (unsigned)sCnt[par][lane] : 0u;
            const int tot = (int)__reduce_add_sync(0xffffffffu, cnt);
            const int off = nq + (int)__reduce_add_sync(0xffffffffu, lane < warp ? cnt : 0u);
            par ^= 1;
            if (queue) sQ[off + __popc(bm & ((1u << lane) - 1u))] = pos;
            nq += tot;
            ++run;
        }
        if (!more || run >= 64) {
            fold_nodes<PREC>(acc0, sF0[warp], lane);
            run = 0;
        }
        if (!more || nq > QCAP - THREADS) {
            __syncthreads();
            if (active) flush(nq);
            __syncthreads();
            nq = 0;
        }
    }
    // ---- Chebyshev coefficients of the node totals, level 0's summed over the warps first
    {
        const bool node = lane < kNodes;
        const float2 f1 = node ? sF1[warp][lane] : make_float2(0.f, 0.f);
        const float c1 = cheb_coefs(f1.x, f1.y, lane);
        if (node) sC1[warp][lane] = c1;
        if (warp == 0) {
            float hi = 0.f, lo = 0.f;
            for (int v = 0; v < WARPS && node; ++v) {
                acc_pair(hi, lo, sF0[v][lane].x);
                lo -= sF0[v][lane].y;
            }
            const float c0 = cheb_coefs(hi, -lo, lane);
            if (node) sC0[lane] = c0;
        }
    }
    __syncthreads();
    const float tp = expf(*g.ln_tp);
    if (active) {
        const float r0 = span0 > 0.f ? 2.f / span0 : 0.f, r1 = span1 > 0.f ? 2.f / span1 : 0.f;
#pragma unroll
        for (int k = 0; k < PTS; ++k) {
            const int j = Js + 32 * k + lane;
            if (k >= npt || j > Je) continue;
            const float near = PREC == MPSA_PREC_FP32_COMPENSATED ? sSum[k][tid] - sComp[k][tid] : sSum[k][tid];
            const float far = clenshaw(sC0, fmaf((float)(j - J0), r0, -1.f)) + clenshaw(sC1[warp], fmaf((float)(j - Js), r1, -1.f));
            g.out[j] = tp * (near + far);
        }
    }
    __syncthreads();   // the shared memory is free for the persistent kernel's next tile
}

// Grid form: one CTA per (row, tile); the rows of one call follow one another in the prep arrays.
struct TileArgs {
    RowDesc row;     // row 0
    size_t ld;       // lines per row of the record array
    int size;        // points of a CTA: a tile, or an even part of one (a multiple of 256)
    int split;       // CTAs per tile at most (1: direct output)
    int split_free;  // as many as the GPU holds at once
    float* part;     // split > 1: partial sums [n_sel][split][N], added by k_split_sum
    int* used;       // split > 1: how many of a tile's CTAs wrote theirs, [n_sel][nT]
};

__device__ __forceinline__ RowDesc row_desc(const TileArgs& g, int s) {
    RowDesc r = g.row;
    r.ln_tp += s;
    r.cum += (size_t)s * kNumClasses * (r.nT + 3);
    r.rec += s * g.ld;
    r.line += s * g.ld;
    r.out += (size_t)s * r.N;
    return r;
}

// CTAs of an SM: 64 registers, or 80 with the wide tile's shared memory (3 CTAs fit)
constexpr int kTilesPerSM = 4, kWidePerSM = 3;
constexpr int kWidePts = 16, kWideTile = kWidePts * kTileThreads;   // 4096 points
// SPLIT: g.split CTAs per tile, each writing its partial sums to g.part (a separate
// instantiation, so that the one-CTA-per-tile form compiles as it would without it).
// PTS: 8, or 16 for the wide tile (tile_size has the rule).
template <int PREC, bool SPLIT, int PTS>
__global__ void __launch_bounds__(kTileThreads, PTS == kWidePts ? kWidePerSM : kTilesPerSM) k_tiles(TileArgs g) {
    RowDesc r = row_desc(g, blockIdx.y);
    if (SPLIT) {
        const int sp = blockIdx.x % g.split;
        r.out = g.part + ((size_t)blockIdx.y * g.split + sp) * r.N;
        const int part = blockIdx.x / g.split, parts = gridDim.x / g.split;
        tile_body<PREC, PTS, kTileThreads>(r, part * g.size, g.size, sp, g.split, g.split_free,
                                           g.used + (size_t)blockIdx.y * parts + part);
    } else {
        tile_body<PREC, PTS, kTileThreads>(r, blockIdx.x * g.size, g.size);
    }
}

// kappa[s][j] = sum over the split CTAs' partial sums (FP64 sum, one rounding to FP32)
__global__ void k_split_sum(int n_sel, int N, int size, int split, const int* __restrict__ used, const float* __restrict__ part,
                            float* __restrict__ kappa) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)n_sel * N) return;
    const int s = (int)(t / N), j = (int)(t % N);
    const int n = used[(size_t)s * ((N + size - 1) / size) + j / size];
    double acc = 0.0;
    for (int q = 0; q < n; ++q) acc += part[((size_t)s * split + q) * N + j];
    kappa[t] = (float)acc;
}

// Persistent form: a fixed grid of CTAs pulls (row, tile) units from a work list
// (ordered by decreasing estimated cost) through one global counter.
template <int PREC, int PTS, int THREADS, int MINB>
__global__ void __launch_bounds__(THREADS, MINB) k_tiles_persistent(const RowDesc* __restrict__ rows,
                                                                   const int2* __restrict__ units, int n_units,
                                                                   int* __restrict__ counter) {
    __shared__ int s_unit;
    for (;;) {
        if (threadIdx.x == 0) s_unit = atomicAdd(counter, 1);
        __syncthreads();
        const int u = s_unit;
        __syncthreads();
        if (u >= n_units) break;
        const int2 rt = units[u];
        const RowDesc r = rows[rt.x];
        tile_body<PREC, PTS, THREADS>(r, rt.y * (PTS * THREADS), PTS * THREADS);
    }
}

// ---------------------------------------------------------------------------
// All-FP64 variant of the profile kernel (precision study): line terms of Eq. (l_nu_line),
// the exact frequency offset v = (c/lambda_j - nu0)/dnuD and H in FP64, plain FP64 sums.
// Same candidate lines and outer windows as the FP32 kernel; the cut threshold is the FP32
// one (t_p = exp(ln t_p)), so inclusion decisions differ only inside the edge slack band.
struct Tile64Args {
    TileArgs t;
    const int* sel;
    const double* pop;
    int pop_stride_;
    int n_sp;
    const int* sp_el;
    const int* sp_stage;
    const double* el;          // [n_el][kElStride] element records
    int n_el;
    double vturb;
    const double* lam_nm;      // line list
    const float* loggf;
    const float* E;
    const float* lgR;
    const float* lgS;
    const float* lgW;
    const int* species;
    double lam0_nm, lnq64;
};

// All-FP64 variant: one point per thread (256-point tiles, so that narrow grids still fill
// the GPU), line constants in FP64 per (line, tile), FP64 Voigt tiers.
constexpr int kTile64 = 256;
__global__ void __launch_bounds__(256) k_tiles64(Tile64Args g) {
    constexpr int THREADS = 256, PTS = 1, TILE = THREADS * PTS;
    static_assert(TILE == kTile64, "FP64 tile size");
    __shared__ double sS[THREADS], sA[THREADS], sNu[THREADS], sDnu[THREADS];
    __shared__ int sLo[THREADS], sHi[THREADS];
    __shared__ int sN;
    const int s = blockIdx.y, tile = blockIdx.x, tid = threadIdx.x;
    const RowDesc r = row_desc(g.t, s);
    const int J0 = tile * TILE;
    const double* row = g.pop + (size_t)(g.sel ? g.sel[s] : s) * g.pop_stride_;
    const double T = row[kPopT], ne = row[kPopNe], nHI = row[kPopNHI], rho = row[kPopRho];
    const double tp = exp((double)*r.ln_tp);
    double nu[PTS], acc[PTS];
    for (int k = 0; k < PTS; ++k) {
        const int j = J0 + k * THREADS + tid;
        nu[k] = kC / (g.lam0_nm * exp((double)j * g.lnq64) * 1e-7);
        acc[k] = 0.0;
    }
    const double pre = sqrt(kPI) * kE * kE / (kME * kC);
    for (int b = 0; b < kNumClasses; ++b) {
        const int reach = 1 << b;
        int tlo = max(floordiv(J0 - reach + 1, TILE), -1), thi = min(floordiv(J0 + TILE - 1 + reach - 1, TILE), r.nT);
        if (tlo > thi) continue;
        const int* cum = r.cum + (size_t)b * (r.nT + 3);
        const int beg = cum[tlo + 1], end = cum[thi + 2];
        for (int base = beg; base < end; base += THREADS) {
            if (tid == 0) sN = 0;
            __syncthreads();
            const int pos = base + tid;
            if (pos < end) {
                const int q = r.line[pos];
                const int jlo = r.rec[pos].jlo, jhi = r.rec[pos].jhi;
                if (jhi >= J0 && jlo <= J0 + TILE - 1) {
                    const int sp = g.species[q];
                    const int e = g.sp_el[sp], st = g.sp_stage[sp];
                    const double lam = g.lam_nm[q] * 1e-7;
                    const double nu0 = kC / lam;
                    const double u = sqrt(2.0 * kKB * T / (g.el[e * kElStride + kElMass] * kAMU) + g.vturb * g.vturb);
                    const double dnu = nu0 * u / kC;
                    const double gam = pow(10.0, (double)g.lgR[q]) + pow(10.0, (double)g.lgS[q]) * ne +
                                       pow(10.0, (double)g.lgW[q]) * nHI;
                    const double NU = row[pop_nu(e, st)];
                    const double S = pre * pow(10.0, (double)g.loggf[q]) * NU / (rho * dnu) *
                                     exp(-(double)g.E[q] * kEV / (kKB * T)) * (-expm1(-kH * nu0 / (kKB * T)));
                    const int slot = atomicAdd(&sN, 1);
                    sS[slot] = S;
                    sA[slot] = gam / (4.0 * kPI * dnu);
                    sNu[slot] = nu0;
                    sDnu[slot] = 1.0 / dnu;
                    sLo[slot] = jlo;
                    sHi[slot] = jhi;
                }
            }
            __syncthreads();
            const int n = sN;
            for (int i = 0; i < n; ++i) {
                const double S = sS[i], a = sA[i], nu0 = sNu[i], inv_dnu = sDnu[i];
                const int lo = sLo[i], hi = sHi[i];
                for (int k = 0; k < PTS; ++k) {
                    const int j = J0 + k * THREADS + tid;
                    if (j < lo || j > hi) continue;
                    const double l = S * voigt_H64((nu[k] - nu0) * inv_dnu, a);
                    if (l >= tp) acc[k] += l;
                }
            }
            __syncthreads();
        }
    }
    for (int k = 0; k < PTS; ++k) {
        const int j = J0 + k * THREADS + tid;
        if (j < r.N) r.out[j] = (float)acc[k];
    }
}

int g_init_mask = 0;

// H in the FP32 form of `which` (mpsa_voigt)
__device__ float voigt_form(float v, float a, int which) {
    const float A = a * a, Z = fmaf(v, v, A);
    if (which == MPSA_VOIGT_CENTRE) return A >= 36.f ? voigt_H(0.f, a) : voigt_core0(a);
    if (which == MPSA_VOIGT_PAIR && A <= kSeriesA && Z >= kSeriesZ2Low && Z <= 1.0e18f)
        return pair_series(make_float2(v, v), A, a * kInvSqrtPi, series_k2(A), series_k3(A), series_k4(A)).x;
    if (which == MPSA_VOIGT_NODE) {
        // every node of the stretch at v; a line that is interpolated passes the cut there, so s_rel (here a
        // power of two) is what makes s_rel H one or more
        const Wing w{v, 0.f, 0.f, Z, Z};
        const float G[kNodes] = {}, ka = a * kInvSqrtPi, srel = exp2f(ceilf(log2f(Z / ka)));
        float2 acc[kNodes / 2] = {};
        if (rational_ok(w, A)) nodes_rational(w, A, srel * ka, G, acc);
        else if (A <= kSeriesA && Z >= kSeriesZ2Low) nodes_series<true>(w, A, srel * ka, G, acc);
        else if (A > kSeriesA && Z >= kSeriesZ2 && Z <= 1.0e18f) nodes_series<false>(w, A, srel * ka, G, acc);
        else return voigt_point(v, a);
        return acc[0].x / srel;
    }
    return which >= MPSA_VOIGT_POINT && which <= MPSA_VOIGT_NODE ? voigt_point(v, a) : voigt_H(v, a);
}

__global__ void k_voigt_eval(int64_t n, const double* __restrict__ v, const double* __restrict__ a, int which,
                             double* __restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = which == MPSA_PREC_FP64 ? voigt_H64(v[i], a[i]) : (double)voigt_form((float)v[i], (float)a[i], which);
}

}  // namespace

int synth_module_init(int device) {
    if (device < 0 || device >= 31) return fail(MPSA_EINVAL, "device %d", device);
    if (g_init_mask & (1 << device)) return MPSA_OK;
    int rc = voigt_upload();
    if (rc != MPSA_OK) return rc;
    g_init_mask |= 1 << device;
    return MPSA_OK;
}

// Shared by synth_opacity and synth_spectrum: synthesis for rows `sel` of a
// population table `pop` onto grid (lam0, R, N); writes kappa [n_sel][N].
// Device buffers of the line preparation of n_sel rows (one grid, one tile size).
struct PrepBufs {
    int64_t L = 0;
    int n_grids = 1;
    size_t ld = 0;   // lines per row of the per-(row, line) arrays: L rounded up to four
    int n_sel = 0, nb = 0;
    int *c = nullptr, *classcnt = nullptr, *line = nullptr;
    LineRec* rec = nullptr;
    float *f = nullptr, *dist = nullptr, *lnS = nullptr, *av = nullptr, *lnk0 = nullptr, *ln_tp = nullptr;
    unsigned char* flag = nullptr;
    RowConst* rc = nullptr;
    SpConst* spc = nullptr;
    MedState* med = nullptr;
    PrepOut po{};
};

// Allocate every prep buffer of n_sel rows on n_grids grids through `al` (stream-ordered scratch or
// persistent memory).
template <class Alloc>
int prep_alloc(PrepBufs& b, const mpsa_ctx* ctx, int n_sel, int n_grids, Alloc&& al) {
    b.L = ctx->L;
    b.n_sel = n_sel;
    b.n_grids = n_grids;
    b.nb = (int)((b.L + kPrepLines - 1) / kPrepLines);
    b.ld = ((size_t)b.L + 3) & ~(size_t)3;
    const size_t GL = n_grids * b.ld, SL = n_sel * b.ld, Sb = (size_t)n_sel * b.nb;
    int r;
    if ((r = al(&b.c, GL)) || (r = al(&b.f, GL)) || (r = al(&b.dist, GL)) || (r = al(&b.flag, GL)) || (r = al(&b.rc, n_sel)) ||
        (r = al(&b.spc, (size_t)n_sel * ctx->n_sp)) || (r = al(&b.lnS, SL)) || (r = al(&b.av, SL)) ||
        (r = al(&b.lnk0, SL)) || (r = al(&b.ln_tp, n_sel)) || (r = al(&b.po.surv, SL)) || (r = al(&b.po.nsurv, n_sel)) ||
        (r = al(&b.po.run, Sb)) || (r = al(&b.po.srel, SL)) || (r = al(&b.po.win, SL)) || (r = al(&b.po.cls, SL)) ||
        (r = al(&b.po.blkcnt, Sb * kNumClasses)) || (r = al(&b.classcnt, (size_t)n_sel * kNumClasses)) || (r = al(&b.rec, SL)) || (r = al(&b.line, SL)) ||
        (r = al(&b.med, n_sel)))
        return r;
    return MPSA_OK;
}

GridDesc grid_desc(double lam0_nm, double lnq, int N, int index) {
    return GridDesc{lam0_nm, lnq, (float)lnq, (float)(1.0 / lam0_nm), (float)(1.0 / (lam0_nm * exp((double)(N - 1) * lnq))),
                    N, index};
}

// Line preparation of the rows d_sel of `pop`: line terms, median continuum and cut threshold, the
// lines that reach the grid, their placement, cut windows and width-class buckets.  One grid for
// all rows (grid), or, with b.n_grids > 1, grid g's descriptor at d_grids[g] and row s's at d_row_grids[s].
int prep_launch(const PrepBufs& b, const mpsa_ctx* ctx, const double* pop, const int* d_sel, const GridDesc& grid,
                const GridDesc* d_grids, const GridDesc* d_row_grids, const RowOut& out, const mpsa_synth_opts* opts,
                cudaStream_t st) {
    const double cut = (opts && opts->cut > 0) ? opts->cut : 1e-3;
    const double kcf = (opts && opts->kc_factor > 0) ? opts->kc_factor : 1e-2;
    const int64_t L = b.L;
    const int n_sel = b.n_sel, n_sp = ctx->n_sp;
    const RowGrids grids{grid, d_row_grids};
    const int pop32 = (opts && opts->precision == MPSA_PREC_FP32_POP32) ? 1 : 0;
    const int cb = (n_sel * n_sp + kStartThreads - 1) / kStartThreads;
    k_start<<<cb + (unsigned)((L + kStartThreads - 1) / kStartThreads), kStartThreads, 0, st>>>(
        cb, n_sel, d_sel, n_sp, ctx->d_sp_el, ctx->d_sp_stage, ctx->n_el, ctx->d_el, pop, ctx->vturb, pop32, b.rc, b.spc,
        b.po.nsurv, L, b.ld, b.n_grids, ctx->d_lam, grid, d_grids, b.dist, b.flag);
    const LineList lines{ctx->d_species, ctx->d_loggf, ctx->d_E, ctx->d_lgR, ctx->d_lgS, ctx->d_lgW, ctx->d_lam};
    int dev = 0, sms = 0;
    MPSA_CUDA_TRY(cudaGetDevice(&dev));
    MPSA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const bool small = L <= kMedSmall;
    // Bounds first, where a grid covers less than a quarter of the list's range: a line that is kept
    // takes its terms after its bounds; and where there are enough pairs to repay two more launches.  80 depths x 5e6
    // lines, 0.2 per cent of the range: 8.80 -> 7.09 ms for the call, 63 depths, 5 per cent: 20.4 -> 19.4 ms; two rows
    // over the whole range 14.0 -> 14.1 ms (so not there); 8 rows x 5e5 lines a call, eight requests at once: 11.4 ->
    // 10.9 ms, 8 x 66,753 lines 4.86 -> 5.04 ms.  Batches always: 8 rows x 1e6 lines on grids over the whole range
    // take 3.95 ms with bounds and 3.93 without, over 41 per cent of it 1.92 and 1.94 ms.
    const bool bounds = !small && (int64_t)n_sel * L >= 3000000 && (d_grids || 4.0 * grid.N * grid.lnq64 < ctx->log_span);
    {
        // ln S, a, ln kappa0 and the median; the record array, not in use yet, holds the listed lines
        // and the sample
        const int rows = (n_sel + kKappa0Rows - 1) / kKappa0Rows;
        const int64_t ns = (L + kMedStride - 1) / kMedStride;
        const size_t ns_ld = ((size_t)ns + 3) & ~(size_t)3;
        float* const list = reinterpret_cast<float*>(b.rec);
        float* const sample = list + (size_t)n_sel * b.ld;
        const unsigned lb = (unsigned)((L + 255) / 256);
        if (!small) {
            k_kappa0<true><<<dim3((unsigned)((ns + 255) / 256), rows), 256, 0, st>>>(L, ns_ld, n_sel, lines, n_sp, b.rc, b.spc,
                                                                                     nullptr, nullptr, sample);
            k_med_bracket<<<n_sel, kMedThreads, 0, st>>>(ns, ns_ld, sample, b.med);
        }
        if (bounds)
            k_bounds<<<dim3(lb, rows), 256, 0, st>>>(L, b.ld, n_sel, lines, n_sp, b.rc, b.spc, b.lnS, b.lnk0);
        else
            k_kappa0<false><<<dim3(lb, rows), 256, 0, st>>>(L, b.ld, n_sel, lines, n_sp, b.rc, b.spc, b.lnS, b.av, b.lnk0);
        if (!small) {
            // eight groups of 128 lines per warp, and no more than four waves of CTAs in all
            const int per_row = (int)std::max<int64_t>(1, std::min<int64_t>(L / 8192, 16ll * sms / n_sel));
            k_med_collect<<<dim3(per_row, n_sel), kCollectThreads, 0, st>>>(L, b.ld, b.lnk0, lines, n_sp, b.rc, b.spc, b.med,
                                                                            list, b.ld);
            if (bounds) k_med_redo<<<dim3(64, n_sel), 256, 0, st>>>(L, b.ld, lines, n_sp, b.rc, b.spc, b.med, b.lnk0);
        }
        k_med_select<<<n_sel, kMedThreads, 0, st>>>(L, b.ld, b.lnk0, small ? nullptr : b.med, list, b.ld,
                                                    (float)log(kcf), (float)log(cut), b.ln_tp, out);
    }
    // up to four blocks of lines per CTA, while 16 CTAs per SM remain (80 rows x 5e6 lines: the call 7.26 ms
    // with one block per CTA, 7.07 with two, 6.99 with four)
    const int gx = (int)std::max<int64_t>((b.nb + 3) / 4, std::min<int64_t>(b.nb, (16 * sms + n_sel - 1) / n_sel));
    auto prep = [&](auto kernel) {
        kernel<<<dim3(gx, n_sel), kPrepThreads, 0, st>>>(L, b.ld, grids, ctx->d_species, b.dist, b.flag, n_sp, b.spc, b.lnS,
                                                           b.av, b.lnk0, b.ln_tp, b.nb, b.po);
    };
    if (bounds) prep(k_prep<true>);
    else prep(k_prep<false>);
    if ((int64_t)b.nb * b.n_grids >= 2 * sms)
        k_place<kPrepLines><<<dim3(b.nb, b.n_grids), kPrepThreads, 0, st>>>(L, b.ld, ctx->d_lam, grid, d_grids, b.flag, b.c,
                                                                            b.f);
    else
        k_place<kPrepThreads><<<dim3((unsigned)((L + kPrepThreads - 1) / kPrepThreads), b.n_grids), kPrepThreads, 0, st>>>(
            L, b.ld, ctx->d_lam, grid, d_grids, b.flag, b.c, b.f);
    {
        // the listed lines' count is known on the device only: about eight CTAs per SM in all,
        // each running over its row's list
        const int gx = std::max(1, std::min(b.nb, (8 * sms + n_sel - 1) / n_sel));
        auto windows = [&](auto kernel) {
            kernel<<<dim3(gx, n_sel), kPrepThreads, 0, st>>>(b.ld, grids, lines, b.c, b.f, n_sp, b.rc, b.spc, b.lnS, b.av,
                                                             b.ln_tp, b.nb, b.po);
        };
        if (bounds) windows(k_windows<true>);
        else windows(k_windows<false>);
    }
    k_scan_class<<<dim3(kNumClasses, n_sel), 1024, 0, st>>>(b.nb, b.po.blkcnt, b.classcnt, out);
    constexpr int kWarps = kPrepThreads / 32;
    if ((int64_t)b.nb * n_sel * kWarps <= 64ll * sms)
        k_scatter<kWarps><<<dim3(b.nb, n_sel), kPrepThreads, 0, st>>>(
            b.ld, grids, ctx->d_species, b.c, b.f, n_sp, b.spc, b.av, b.po.blkcnt, b.classcnt, b.nb, b.po, b.rec,
            b.line, out);
    else
        k_scatter<1><<<dim3((b.nb + kWarps - 1) / kWarps, n_sel), kPrepThreads, 0, st>>>(
            b.ld, grids, ctx->d_species, b.c, b.f, n_sp, b.spc, b.av, b.po.blkcnt, b.classcnt, b.nb, b.po, b.rec,
            b.line, out);
    MPSA_CUDA_TRY(cudaGetLastError());
    return MPSA_OK;
}

// Tile ranges of all rows for the descriptors (see k_ranges); most: the largest number of tiles.
int ranges_launch(const PrepBufs& b, const RowDesc& one, const RowDesc* d_rows, int most, cudaStream_t st) {
    const int n = kNumClasses * (most + 3);
    k_ranges<<<dim3((n + 255) / 256, b.n_sel), 256, 0, st>>>(b.n_sel, b.ld, one, d_rows, b.classcnt);
    MPSA_CUDA_TRY(cudaGetLastError());
    return MPSA_OK;
}

// A row on a grid for tiles of `tile` points: its tile ranges, output, cut threshold and records.
RowDesc row_of(const GridDesc& q, int tile, int* cum, const float* ln_tp, const LineRec* rec, const int* line, float* out) {
    RowDesc r;
    r.N = q.N;
    r.nT = (q.N + tile - 1) / tile;
    r.tile = tile;
    r.lnq = q.lnq;
    r.q1 = (float)(-q.lnq64 / 2.0);
    r.q2 = (float)(q.lnq64 * q.lnq64 / 6.0);
    r.ln_tp = ln_tp;
    r.cum = cum;
    r.rec = rec;
    r.line = line;
    r.out = out;
    return r;
}

// Points per tile.  Level 0 works through a tile's candidate lines once, so a tile of twice the points halves
// it, and the tile's fixed cost; but the parts of its warps are twice as long as well, and a line
// near a part costs an evaluation at each of its points.  Windows are wider in grid points on finer
// grids, and few lines leave the fixed cost: 4096 points from R = 1e6 on, or below one line in 20
// points of the list's range, if these tiles fill the GPU.  2048 -> 4096 points, whole calls: two rows
// of 5e6 lines, 300 - 1500 nm, at R = 2e6 4829 -> 4178 us, 1e6 3767 -> 3562, 5e5 3316 -> 3304 and 2e5
// 2726 -> 3665 us; eight rows at R = 5e5 with 1.5e6 lines 5220 -> 6003 us, 5e5 lines 2120 -> 2156, 1e5
// lines 712 -> 651 us.
int tile_size(const mpsa_ctx* ctx, int n_sel, int N, double R, int sms) {
    const bool fine = R >= 1e6, sparse = (double)ctx->L * 20.0 < ctx->log_span * R;
    const int64_t wide = (int64_t)((N + kWideTile - 1) / kWideTile) * n_sel;
    return (fine || sparse) && wide >= (int64_t)kWidePerSM * sms ? kWideTile : kTile;
}

// A call with fewer tiles than the GPU holds CTAs (narrow windows) shares each tile out:
//  * of lists up to 1e5 lines, by points, down to 256 a CTA, while half the GPU stays free: near lines are
//    evaluated point by point, and a shorter part has fewer of them.  Every CTA runs over the
//    tile's candidates, which costs more the longer the list is.  The call without and with it, us, 40 rows of
//    2000 points: 20,000 lines 561 and 343, 100,000 lines 1352 and 930, 300,000 lines 2326 and 1738; of 500
//    points: 300 and 289, 658 and 656, 1122 and 1212 (150,000 lines 756 and 782);
//  * of lists above 2048 lines, by candidate lines, over up to 64 CTAs, with partial sums added afterwards: as
//    many as run at once, one chunk each at least, and up to eight times that for
//    the tiles with kSplitChunks each (deep rows have ten times the candidates of shallow ones).
//    Shorter lists save the second kernel.  With and without, us, 4 rows of 8000 points: 300 lines 151 and 115, 2048
//    lines 173 and 134, 5000 lines 185 and 147, 10,000 lines 191 and 162; 40 rows: 189 and 152, 256 and 234, 329 and
//    338, 428 and 481 (the line lies on the safe side of the two).
// peers: calls that run beside this one take their part of the GPU.  Eight spectrum requests at once on eight
// streams: 12.8 ms when each counts on the whole GPU, 11.5 ms on an eighth; seven on 25,000 lines 5.6, 3.7 ms.
void tile_split(TileArgs& ta, int tile, int n_sel, int N, int64_t L, int sms, int peers) {
    const int64_t slots = (int64_t)sms * kTilesPerSM / peers;
    auto ctas = [&](int size) { return (int64_t)((N + size - 1) / size) * n_sel; };
    ta.size = tile;
    while (tile == kTile && L <= 100000 && ta.size > 256 && 2 * ctas(ta.size / 2) <= slots) ta.size /= 2;
    const int64_t n = ctas(ta.size), most = std::min<int64_t>(64, kNumClasses + L / kTileThreads);   // chunks a tile can have
    ta.split_free = (int)std::max<int64_t>(1, std::min(most, slots / n));
    ta.split = tile != kTile || L <= 2048 || n > slots ? 1 : (int)std::max<int64_t>(1, std::min(most, 8 * slots / n));
    ta.part = nullptr;
    ta.used = nullptr;
}

// The scratch of one synth_rows call: its arrays, added to one block.
struct SynthScratch {
    PrepBufs b;
    TileArgs ta;
    int *cum = nullptr, tile = 0, nT = 0, nC = 0;   // nC: CTAs of a row, before the split by candidates
    ScratchBlock block;
    SynthScratch(const mpsa_ctx* ctx, int n_sel, int N, double R, int prec, int sms, int peers) {
        tile = prec == MPSA_PREC_FP64 ? kTile64 : tile_size(ctx, n_sel, N, R, sms);
        nT = (N + tile - 1) / tile;
        prep_alloc(b, ctx, n_sel, 1, [&](auto** p, size_t n) { return block.add(p, n); });
        block.add(&cum, (size_t)n_sel * kNumClasses * (nT + 3));
        tile_split(ta, tile, n_sel, N, b.L, sms, peers);
        nC = (N + ta.size - 1) / ta.size;
        if (ta.split > 1) {
            block.add(&ta.part, (size_t)n_sel * ta.split * N);
            block.add(&ta.used, (size_t)n_sel * nC);
        }
    }
};

size_t synth_rows_bytes(const mpsa_ctx* ctx, int n_sel, int N, double R, int peers) {
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device) != cudaSuccess) sms = 1;
    return SynthScratch(ctx, n_sel, N, R, MPSA_PREC_FP32_COMPENSATED, sms, peers).block.bytes;
}

int synth_rows(mpsa_ctx* ctx, const double* pop, int n_sel, const int* d_sel, double lam0_nm, double R, int N,
               float* kappa, float* kc_out, int64_t* evals, const mpsa_synth_opts* opts, cudaStream_t st, int peers) {
    const int prec = opts ? opts->precision : 0;
    if (prec != MPSA_PREC_FP32_COMPENSATED && prec != MPSA_PREC_FP32_NAIVE && prec != MPSA_PREC_FP64 &&
        prec != MPSA_PREC_FP32_POP32)
        return fail(MPSA_EINVAL, "synth: precision %d", prec);
    Scratch sc(st, ctx->pool);
    int r, dev = 0, sms = 0;
    MPSA_CUDA_TRY(cudaGetDevice(&dev));
    MPSA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    SynthScratch scratch(ctx, n_sel, N, R, prec, sms, peers);
    if ((r = scratch.block.take(sc))) return r;
    PrepBufs& b = scratch.b;
    TileArgs& ta = scratch.ta;
    int* const cum = scratch.cum;
    const int tile = scratch.tile, nT = scratch.nT, nC = scratch.nC;
    const GridDesc grid = grid_desc(lam0_nm, log1p(1.0 / R), N, 0);
    const RowOut out{kc_out, (unsigned long long*)evals, nullptr, nullptr};
    if ((r = prep_launch(b, ctx, pop, d_sel, grid, nullptr, nullptr, out, opts, st))) return r;
    ta.row = row_of(grid, tile, cum, b.ln_tp, b.rec, b.line, kappa);
    ta.ld = b.ld;
    if ((r = ranges_launch(b, ta.row, nullptr, nT, st))) return r;
    prof_mark(ctx, MPSA_KERNEL_PROFILE, st);
    if (prec == MPSA_PREC_FP64) {
        Tile64Args g;
        g.t = ta;
        g.sel = d_sel;
        g.pop = pop;
        g.pop_stride_ = pop_stride(ctx->n_el);
        g.n_sp = ctx->n_sp;
        g.sp_el = ctx->d_sp_el;
        g.sp_stage = ctx->d_sp_stage;
        g.el = ctx->d_el;
        g.n_el = ctx->n_el;
        g.vturb = ctx->vturb;
        g.lam_nm = ctx->d_lam;
        g.loggf = ctx->d_loggf;
        g.E = ctx->d_E;
        g.lgR = ctx->d_lgR;
        g.lgS = ctx->d_lgS;
        g.lgW = ctx->d_lgW;
        g.species = ctx->d_species;
        g.lam0_nm = lam0_nm;
        g.lnq64 = grid.lnq64;
        k_tiles64<<<dim3(nT, n_sel), 256, 0, st>>>(g);
    } else {
        const dim3 blocks((unsigned)(nC * ta.split), n_sel);
        auto go = [&](auto kernel) { kernel<<<blocks, kTileThreads, 0, st>>>(ta); };
        const bool naive = prec == MPSA_PREC_FP32_NAIVE;
        if (tile == kWideTile) {
            if (naive) go(k_tiles<MPSA_PREC_FP32_NAIVE, false, kWidePts>);
            else go(k_tiles<MPSA_PREC_FP32_COMPENSATED, false, kWidePts>);
        } else if (ta.split > 1) {
            if (naive) go(k_tiles<MPSA_PREC_FP32_NAIVE, true, kPtsPerThread>);
            else go(k_tiles<MPSA_PREC_FP32_COMPENSATED, true, kPtsPerThread>);
        } else {
            if (naive) go(k_tiles<MPSA_PREC_FP32_NAIVE, false, kPtsPerThread>);
            else go(k_tiles<MPSA_PREC_FP32_COMPENSATED, false, kPtsPerThread>);
        }
        if (ta.split > 1) {
            const int64_t tot = (int64_t)n_sel * N;
            k_split_sum<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(n_sel, N, ta.size, ta.split, ta.used, ta.part, kappa);
        }
    }
    prof_mark(ctx, MPSA_KERNEL_PROFILE, st);
    MPSA_CUDA_TRY(cudaGetLastError());
    return MPSA_OK;
}

int check_species(const mpsa_ctx* ctx, const char* who) {
    for (int i = 0; i < ctx->n_sp; ++i) {
        const int e = ctx->h_sp_el[i], st = ctx->h_sp_stage[i];
        if (e >= ctx->n_el) return fail(MPSA_EINVAL, "%s: species %d refers to element %d of %d", who, i, e, ctx->n_el);
        if (st >= (int)ctx->h_el[(size_t)e * kElStride + kElStages])
            return fail(MPSA_EINVAL, "%s: species %d is stage %d of element %d, which has %d stages", who, i, st, e,
                        (int)ctx->h_el[(size_t)e * kElStride + kElStages]);
    }
    return MPSA_OK;
}

int check_grid(const mpsa_lgrid* g, int* N) {
    const int64_t n = mpsa_grid_size(g);
    if (n < 1) return fail(MPSA_EINVAL, "invalid grid");
    if (n >= kMaxGrid - kTile) return fail(MPSA_EINVAL, "grid of %lld points exceeds %d", (long long)n, kMaxGrid - kTile);
    *N = (int)n;
    return MPSA_OK;
}

}  // namespace mpsa

using namespace mpsa;

extern "C" int synth_opacity(mpsa_ctx* ctx, const mpsa_lgrid* grid, int32_t n_sel, const int32_t* sel,
                             float* kappa_out, float* kappa_c_out, int64_t* evals_out, const mpsa_synth_opts* opts,
                             void* stream) {
    if (!ctx || !grid || !sel || !kappa_out) return fail(MPSA_EINVAL, "synth_opacity: NULL argument");
    if (ctx->L < 1 || ctx->n_sp < 1) return fail(MPSA_ESTATE, "synth_opacity: no line list loaded");
    if (!ctx->d_pop) return fail(MPSA_ESTATE, "synth_opacity: no atmosphere grid set");
    if (n_sel < 1) return fail(MPSA_EINVAL, "synth_opacity: n_sel = %d", n_sel);
    int N, r;
    if ((r = check_species(ctx, "synth_opacity"))) return r;
    const int rows = ctx->n_comp * ctx->n_points;
    for (int i = 0; i < n_sel; ++i)
        if (sel[i] < 0 || sel[i] >= rows) return fail(MPSA_EINVAL, "synth_opacity: sel[%d] = %d of %d rows", i, sel[i], rows);
    if ((r = check_grid(grid, &N))) return r;
    if ((size_t)n_sel * ctx->L >= (size_t)1 << 31)
        return fail(MPSA_EINVAL, "synth_opacity: n_sel * n_lines must stay below 2^31 (split the rows)");
    MPSA_CUDA_TRY(cudaSetDevice(ctx->device));
    cudaStream_t st = (cudaStream_t)stream;
    int* d_sel;
    {
        Scratch s2(st, ctx->pool);
        if ((r = s2.alloc(&d_sel, n_sel))) return r;
        MPSA_CUDA_TRY(cudaMemcpyAsync(d_sel, sel, n_sel * sizeof(int), cudaMemcpyHostToDevice, st));
        r = synth_rows(ctx, ctx->d_pop, n_sel, d_sel, grid->lambda0_nm, grid->R, N, kappa_out, kappa_c_out, evals_out,
                       opts, st);
    }
    return r;
}

// ===========================================================================
// Batched form: many rows on several grids in one persistent, graph-captured launch.
//
// At creation every group's line preparation runs once; an autotuner times the
// persistent profile kernel for each candidate (points per thread, threads per CTA,
// CTAs per SM) on a sample of tiles and keeps the fastest per grid point; the
// (row, tile) work units are ordered by decreasing estimated cost (candidate lines
// per tile, largest first); then the whole pipeline (preparation of every group,
// one persistent profile launch over all units, the ODFs) is captured into a CUDA
// graph that mpsa_batch_run replays.
namespace mpsa {
namespace {

struct TuneCfg {
    int pts, threads, minb;
};
constexpr TuneCfg kCfgs[] = {{8, 256, 4}, {4, 256, 4}, {8, 128, 8}, {16, 256, 3}};
constexpr int kNumCfgs = sizeof(kCfgs) / sizeof(kCfgs[0]);

template <int PREC, int PTS, int THREADS, int MINB>
int persistent_launch_t(const RowDesc* rows, const int2* units, int n_units, int* counter, cudaStream_t st) {
    int dev = 0, sms = 0, per_sm = 0;
    MPSA_CUDA_TRY(cudaGetDevice(&dev));
    MPSA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    MPSA_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tiles_persistent<PREC, PTS, THREADS, MINB>,
                                                                THREADS, 0));
    const int grid = std::max(1, std::min(n_units, sms * std::max(per_sm, 1)));
    k_tiles_persistent<PREC, PTS, THREADS, MINB><<<grid, THREADS, 0, st>>>(rows, units, n_units, counter);
    MPSA_CUDA_TRY(cudaGetLastError());
    return MPSA_OK;
}

int persistent_launch(int cfg, int prec, const RowDesc* rows, const int2* units, int n_units, int* counter,
                      cudaStream_t st) {
    MPSA_CUDA_TRY(cudaMemsetAsync(counter, 0, sizeof(int), st));
    if (prec == MPSA_PREC_FP32_NAIVE) {
        switch (cfg) {
            case 0: return persistent_launch_t<1, 8, 256, 4>(rows, units, n_units, counter, st);
            case 1: return persistent_launch_t<1, 4, 256, 4>(rows, units, n_units, counter, st);
            case 2: return persistent_launch_t<1, 8, 128, 8>(rows, units, n_units, counter, st);
            default: return persistent_launch_t<1, 16, 256, 3>(rows, units, n_units, counter, st);
        }
    }
    switch (cfg) {
        case 0: return persistent_launch_t<0, 8, 256, 4>(rows, units, n_units, counter, st);
        case 1: return persistent_launch_t<0, 4, 256, 4>(rows, units, n_units, counter, st);
        case 2: return persistent_launch_t<0, 8, 128, 8>(rows, units, n_units, counter, st);
        default: return persistent_launch_t<0, 16, 256, 3>(rows, units, n_units, counter, st);
    }
}

// Estimated cost of a (row, tile) unit: the number of candidate lines of the tile.
__global__ void k_unit_cost(const RowDesc* __restrict__ rows, const int2* __restrict__ units, int n_units,
                            long long* __restrict__ cost) {
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= n_units) return;
    const int2 rt = units[u];
    const RowDesc r = rows[rt.x];
    const int TILE = r.tile, J0 = rt.y * TILE;
    long long n = 0;
    for (int b = 0; b < kNumClasses; ++b) {
        const int reach = 1 << b;
        int tlo = max(floordiv(J0 - reach + 1, TILE), -1), thi = min(floordiv(J0 + TILE - 1 + reach - 1, TILE), r.nT);
        if (tlo > thi) continue;
        const int* cum = r.cum + (size_t)b * (r.nT + 3);
        n += cum[thi + 2] - cum[tlo + 1];
    }
    cost[u] = n;
}

}  // namespace
}  // namespace mpsa

struct mpsa_batch {
    mpsa_ctx* ctx = nullptr;
    mpsa_synth_opts opts{};
    int prec = 0, cfg = 0;
    struct Group {
        mpsa_lgrid grid{};
        int N = 0, n_sel = 0;
        int part = 0, row0 = 0;   // its rows' place in a part
        mpsa::GridDesc q{};
        const int32_t* sel = nullptr;   // host, during creation only
        float *kappa = nullptr, *kc = nullptr;
        int64_t* evals = nullptr;
        int K = 0, n_steps = 0, mean_kind = MPSA_MEAN_ARITH;
        int64_t* d_bounds = nullptr;
        double *d_cw = nullptr, *d_w = nullptr, *odf = nullptr;
        int64_t longest = 0;
    };
    std::vector<Group> groups;
    // consecutive groups whose rows are prepared together (one launch per kernel, not one per group)
    struct Part {
        int n_rows = 0, n_grids = 0, row0 = 0;   // row0: its first row among all
        mpsa::PrepBufs pb;
        int* d_sel = nullptr;
        mpsa::GridDesc *d_grids = nullptr, *d_row_grids = nullptr;
        mpsa::RowOut out{};
    };
    std::vector<Part> parts;
    mpsa::RowDesc* d_rows = nullptr;
    int n_rows = 0;
    int2* d_units = nullptr;
    int n_units = 0;
    int* d_counter = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    std::vector<void*> allocs;
    double tune_ms_per_mpt[mpsa::kNumCfgs] = {0};
    int n_tuned = 0;
};

namespace mpsa {
namespace {

template <class T>
int balloc(mpsa_batch* b, T** p, size_t n) {
    void* q = nullptr;
    cudaError_t e = cudaMalloc(&q, n * sizeof(T) + 16);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(MPSA_ENOMEM, "mpsa_batch_create: cudaMalloc(%zu): %s", n * sizeof(T), cudaGetErrorString(e));
    }
    b->allocs.push_back(q);
    *p = static_cast<T*>(q);
    return MPSA_OK;
}

// Row descriptors of every row of every group for tiles of `tile` points, with a new array of tile
// ranges, on the device; the tile ranges themselves by batch_ranges.
int batch_rows(mpsa_batch* b, int tile, std::vector<RowDesc>* rows) {
    size_t n = 0;
    for (auto& G : b->groups) n += (size_t)G.n_sel * kNumClasses * ((G.N + tile - 1) / tile + 3);
    int r, *cum;
    if ((r = balloc(b, &cum, n))) return r;
    rows->clear();
    for (auto& G : b->groups) {
        const PrepBufs& pb = b->parts[G.part].pb;
        for (int s = 0; s < G.n_sel; ++s) {
            rows->push_back(row_of(G.q, tile, cum, pb.ln_tp + G.row0 + s, pb.rec + (G.row0 + s) * pb.ld,
                                   pb.line + (G.row0 + s) * pb.ld, G.kappa + (size_t)s * G.N));
            cum += (size_t)kNumClasses * (rows->back().nT + 3);
        }
    }
    MPSA_CUDA_TRY(cudaMemcpy(b->d_rows, rows->data(), rows->size() * sizeof(RowDesc), cudaMemcpyHostToDevice));
    return MPSA_OK;
}

int batch_ranges(const mpsa_batch* b, int tile, cudaStream_t st) {
    for (auto& P : b->parts) {
        int most = 0, r;
        for (auto& G : b->groups)
            if (&b->parts[G.part] == &P) most = std::max(most, (G.N + tile - 1) / tile);
        if ((r = ranges_launch(P.pb, RowDesc{}, b->d_rows + P.row0, most, st))) return r;
    }
    return MPSA_OK;
}

int batch_prep(const mpsa_batch* b, cudaStream_t st) {
    for (auto& P : b->parts) {
        const int r = prep_launch(P.pb, b->ctx, b->ctx->d_pop, P.d_sel, GridDesc{}, P.d_grids, P.d_row_grids, P.out, &b->opts,
                                  st);
        if (r) return r;
    }
    return MPSA_OK;
}

constexpr int kPartRows = 32768;   // rows of one preparation (the y dimension of its launches)

int batch_build(mpsa_batch* b, const mpsa_batch_group* gin, int n_groups, int autotune, cudaStream_t st) {
    mpsa_ctx* c = b->ctx;
    int r;
    // ---- groups: grids, rows, persistent prep buffers, ODF parameters
    for (int g = 0; g < n_groups; ++g) {
        const mpsa_batch_group& q = gin[g];
        mpsa_batch::Group G;
        G.grid = q.grid;
        if ((r = check_grid(&q.grid, &G.N))) return r;
        if (q.n_sel < 1 || !q.sel || !q.kappa_out) return fail(MPSA_EINVAL, "mpsa_batch_create: group %d rows/outputs", g);
        const int rows = c->n_comp * c->n_points;
        for (int i = 0; i < q.n_sel; ++i)
            if (q.sel[i] < 0 || q.sel[i] >= rows) return fail(MPSA_EINVAL, "mpsa_batch_create: group %d sel[%d]", g, i);
        if ((size_t)q.n_sel * c->L >= (size_t)1 << 31) return fail(MPSA_EINVAL, "mpsa_batch_create: group %d too large", g);
        G.n_sel = q.n_sel;
        G.kappa = q.kappa_out;
        G.kc = q.kappa_c_out;
        G.evals = q.evals_out;
        G.sel = q.sel;
        if (b->parts.empty() || b->parts.back().n_rows + q.n_sel > kPartRows) {
            b->parts.emplace_back();
            b->parts.back().row0 = b->n_rows;
        }
        mpsa_batch::Part& P = b->parts.back();
        G.part = (int)b->parts.size() - 1;
        G.row0 = P.n_rows;
        G.q = grid_desc(q.grid.lambda0_nm, log1p(1.0 / q.grid.R), G.N, P.n_grids);
        P.n_rows += q.n_sel;
        ++P.n_grids;
        if (q.K > 0) {
            if (!q.bounds || !q.widths || !q.odf_out) return fail(MPSA_EINVAL, "mpsa_batch_create: group %d ODF args", g);
            std::vector<double> cw(q.n_steps >= 1 && q.n_steps <= 32 ? q.n_steps + 1 : 1);
            if ((r = odf_check("mpsa_batch_create", q.n_sel, G.N, q.K, q.bounds, q.n_steps, q.widths, q.mean_kind,
                               cw.data())))
                return r;
            G.K = q.K;
            G.n_steps = q.n_steps;
            G.mean_kind = q.mean_kind;
            G.odf = q.odf_out;
            G.longest = odf_longest(q.K, q.bounds);
            if ((r = balloc(b, &G.d_bounds, q.K + 1)) || (r = balloc(b, &G.d_cw, q.n_steps + 1)) ||
                (r = balloc(b, &G.d_w, q.n_steps)))
                return r;
            MPSA_CUDA_TRY(cudaMemcpy(G.d_bounds, q.bounds, (q.K + 1) * sizeof(int64_t), cudaMemcpyHostToDevice));
            MPSA_CUDA_TRY(cudaMemcpy(G.d_cw, cw.data(), (q.n_steps + 1) * sizeof(double), cudaMemcpyHostToDevice));
            MPSA_CUDA_TRY(cudaMemcpy(G.d_w, q.widths, q.n_steps * sizeof(double), cudaMemcpyHostToDevice));
        }
        b->groups.push_back(G);
        b->n_rows += q.n_sel;
    }
    // ---- parts: buffers, rows, grids and output pointers
    for (size_t p = 0; p < b->parts.size(); ++p) {
        mpsa_batch::Part& P = b->parts[p];
        if ((r = prep_alloc(P.pb, c, P.n_rows, P.n_grids, [&](auto** q, size_t n) { return balloc(b, q, n); }))) return r;
        std::vector<int> sel;
        std::vector<GridDesc> grids, row_grids;
        std::vector<float*> kc;
        std::vector<unsigned long long*> ev;
        for (auto& G : b->groups) {
            if (G.part != (int)p) continue;
            grids.push_back(G.q);
            for (int s = 0; s < G.n_sel; ++s) {
                sel.push_back(G.sel[s]);
                row_grids.push_back(G.q);
                kc.push_back(G.kc ? G.kc + s : nullptr);
                ev.push_back(G.evals ? (unsigned long long*)G.evals + s : nullptr);
            }
            G.sel = nullptr;
        }
        float** d_kc;
        unsigned long long** d_ev;
        if ((r = balloc(b, &P.d_sel, sel.size())) || (r = balloc(b, &P.d_grids, grids.size())) ||
            (r = balloc(b, &P.d_row_grids, sel.size())) || (r = balloc(b, &d_kc, sel.size())) ||
            (r = balloc(b, &d_ev, sel.size())))
            return r;
        MPSA_CUDA_TRY(cudaMemcpy(P.d_sel, sel.data(), sel.size() * sizeof(int), cudaMemcpyHostToDevice));
        MPSA_CUDA_TRY(cudaMemcpy(P.d_grids, grids.data(), grids.size() * sizeof(GridDesc), cudaMemcpyHostToDevice));
        MPSA_CUDA_TRY(cudaMemcpy(P.d_row_grids, row_grids.data(), sel.size() * sizeof(GridDesc), cudaMemcpyHostToDevice));
        MPSA_CUDA_TRY(cudaMemcpy(d_kc, kc.data(), sel.size() * sizeof(float*), cudaMemcpyHostToDevice));
        MPSA_CUDA_TRY(cudaMemcpy(d_ev, ev.data(), sel.size() * sizeof(unsigned long long*), cudaMemcpyHostToDevice));
        P.out = RowOut{nullptr, nullptr, d_kc, d_ev};
    }
    if ((r = batch_prep(b, st))) return r;
    MPSA_CUDA_TRY(cudaStreamSynchronize(st));
    if ((r = balloc(b, &b->d_rows, b->n_rows)) || (r = balloc(b, &b->d_counter, 1))) return r;

    // ---- autotune: time per grid point of each configuration on a sample of tiles
    b->cfg = 0;
    if (autotune) {
        cudaEvent_t e0, e1;
        MPSA_CUDA_TRY(cudaEventCreate(&e0));
        MPSA_CUDA_TRY(cudaEventCreate(&e1));
        double best = 1e300;
        for (int k = 0; k < kNumCfgs; ++k) {
            const int tile = kCfgs[k].pts * kCfgs[k].threads;
            std::vector<RowDesc> rows;
            if ((r = batch_rows(b, tile, &rows)) || (r = batch_ranges(b, tile, st))) return r;
            // sample: at least 2048 (row, tile) units (all of them if there are fewer) spread
            // evenly over all units of the batch, so that rows weigh by their tile counts as in
            // the real launch and every CTA of the persistent launch runs several units (the
            // time then measures throughput, not the slowest unit)
            std::vector<int2> all;
            for (int i = 0; i < (int)rows.size(); ++i)
                for (int t = 0; t < rows[i].nT; ++t) all.push_back(make_int2(i, t));
            std::vector<int2> units;
            const size_t step = std::max<size_t>(1, all.size() / 2048);
            for (size_t u = step / 2; u < all.size(); u += step) units.push_back(all[u]);
            int2* du;
            if ((r = balloc(b, &du, units.size()))) return r;
            MPSA_CUDA_TRY(cudaMemcpy(du, units.data(), units.size() * sizeof(int2), cudaMemcpyHostToDevice));
            float ms_best = 1e30f;
            for (int rep = 0; rep < 2; ++rep) {
                MPSA_CUDA_TRY(cudaEventRecord(e0, st));
                if ((r = persistent_launch(k, b->prec, b->d_rows, du, (int)units.size(), b->d_counter, st))) return r;
                MPSA_CUDA_TRY(cudaEventRecord(e1, st));
                MPSA_CUDA_TRY(cudaEventSynchronize(e1));
                float ms = 0.f;
                MPSA_CUDA_TRY(cudaEventElapsedTime(&ms, e0, e1));
                ms_best = std::min(ms_best, ms);
            }
            const double per_mpt = ms_best / ((double)units.size() * tile / 1e6);
            b->tune_ms_per_mpt[k] = per_mpt;
            if (per_mpt < best) {
                best = per_mpt;
                b->cfg = k;
            }
        }
        b->n_tuned = kNumCfgs;
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
    }

    // ---- final tile ranges, row descriptors and the cost-ordered work list
    const int tile = kCfgs[b->cfg].pts * kCfgs[b->cfg].threads;
    std::vector<RowDesc> rows;
    MPSA_CUDA_TRY(cudaStreamSynchronize(st));   // the descriptors of the last trial are overwritten
    if ((r = batch_rows(b, tile, &rows)) || (r = batch_ranges(b, tile, st))) return r;
    std::vector<int2> units;
    for (int i = 0; i < (int)rows.size(); ++i)
        for (int t = 0; t < rows[i].nT; ++t) units.push_back(make_int2(i, t));
    b->n_units = (int)units.size();
    if ((r = balloc(b, &b->d_units, units.size()))) return r;
    long long* dcost;
    if ((r = balloc(b, &dcost, units.size()))) return r;
    MPSA_CUDA_TRY(cudaMemcpy(b->d_units, units.data(), units.size() * sizeof(int2), cudaMemcpyHostToDevice));
    MPSA_CUDA_TRY(cudaStreamSynchronize(st));
    k_unit_cost<<<(b->n_units + 255) / 256, 256, 0, st>>>(b->d_rows, b->d_units, b->n_units, dcost);
    MPSA_CUDA_TRY(cudaGetLastError());
    std::vector<long long> cost(units.size());
    MPSA_CUDA_TRY(cudaMemcpyAsync(cost.data(), dcost, cost.size() * sizeof(long long), cudaMemcpyDeviceToHost, st));
    MPSA_CUDA_TRY(cudaStreamSynchronize(st));
    std::vector<int> order(units.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return cost[x] > cost[y]; });
    std::vector<int2> sorted(units.size());
    for (size_t i = 0; i < order.size(); ++i) sorted[i] = units[order[i]];
    MPSA_CUDA_TRY(cudaMemcpy(b->d_units, sorted.data(), sorted.size() * sizeof(int2), cudaMemcpyHostToDevice));

    // ---- capture the pipeline into a CUDA graph
    if ((r = odf_setup())) return r;
    cudaStream_t cap;
    MPSA_CUDA_TRY(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
    cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) {
        cudaStreamDestroy(cap);
        return fail(MPSA_ECUDA, "mpsa_batch_create: begin capture: %s", cudaGetErrorString(e));
    }
    int rc = MPSA_OK;
    if ((rc = batch_prep(b, cap)) == MPSA_OK) rc = batch_ranges(b, tile, cap);
    if (rc == MPSA_OK) rc = persistent_launch(b->cfg, b->prec, b->d_rows, b->d_units, b->n_units, b->d_counter, cap);
    if (rc == MPSA_OK)
        for (auto& G : b->groups)
            if (G.K > 0 && (rc = odf_launch(G.kappa, G.n_sel, G.N, G.K, G.d_bounds, G.n_steps, G.d_cw, G.d_w, G.odf, G.mean_kind, G.longest, cap)))
                break;
    e = cudaStreamEndCapture(cap, &b->graph);
    cudaStreamDestroy(cap);
    if (rc != MPSA_OK) return rc;
    if (e != cudaSuccess) return fail(MPSA_ECUDA, "mpsa_batch_create: end capture: %s", cudaGetErrorString(e));
    MPSA_CUDA_TRY(cudaGraphInstantiate(&b->exec, b->graph, 0));
    return MPSA_OK;
}

}  // namespace
}  // namespace mpsa

extern "C" {

int mpsa_batch_create(mpsa_ctx* ctx, int32_t n_groups, const mpsa_batch_group* groups, const mpsa_synth_opts* opts,
                      int32_t autotune, void* stream, mpsa_batch** out) {
    if (!ctx || !groups || !out || n_groups < 1) return fail(MPSA_EINVAL, "mpsa_batch_create: bad argument");
    if (ctx->L < 1 || !ctx->d_pop) return fail(MPSA_ESTATE, "mpsa_batch_create: load a line list and a grid first");
    int rs;
    if ((rs = check_species(ctx, "mpsa_batch_create"))) return rs;
    const int prec = opts ? opts->precision : 0;
    if (prec != MPSA_PREC_FP32_COMPENSATED && prec != MPSA_PREC_FP32_NAIVE)
        return fail(MPSA_EINVAL, "mpsa_batch_create: precision %d", prec);
    MPSA_CUDA_TRY(cudaSetDevice(ctx->device));
    *out = nullptr;
    mpsa_batch* b = new mpsa_batch();
    b->ctx = ctx;
    if (opts) b->opts = *opts;
    b->prec = prec;
    const int r = batch_build(b, groups, n_groups, autotune, (cudaStream_t)stream);
    if (r != MPSA_OK) {
        mpsa_batch_destroy(b);
        return r;
    }
    *out = b;
    return MPSA_OK;
}

int mpsa_batch_run(mpsa_batch* b, void* stream) {
    if (!b || !b->exec) return fail(MPSA_EINVAL, "mpsa_batch_run: bad batch");
    MPSA_CUDA_TRY(cudaSetDevice(b->ctx->device));
    prof_mark(b->ctx, MPSA_KERNEL_PROFILE, (cudaStream_t)stream);
    MPSA_CUDA_TRY(cudaGraphLaunch(b->exec, (cudaStream_t)stream));
    prof_mark(b->ctx, MPSA_KERNEL_PROFILE, (cudaStream_t)stream);
    return MPSA_OK;
}

int mpsa_batch_get_info(const mpsa_batch* b, mpsa_batch_info* out) {
    if (!b || !out) return fail(MPSA_EINVAL, "mpsa_batch_get_info: bad argument");
    out->pts_per_thread = kCfgs[b->cfg].pts;
    out->threads = kCfgs[b->cfg].threads;
    out->min_blocks = kCfgs[b->cfg].minb;
    out->n_rows = b->n_rows;
    out->n_units = b->n_units;
    out->n_tuned = b->n_tuned;
    for (int k = 0; k < 8; ++k) out->tune_ms_per_mpoint[k] = k < kNumCfgs ? b->tune_ms_per_mpt[k] : 0.0;
    return MPSA_OK;
}

int mpsa_voigt(mpsa_ctx* ctx, const double* v, const double* a, int64_t n, int32_t precision, double* out,
               void* stream) {
    if (!ctx || n < 0 || (n > 0 && (!v || !a || !out))) return fail(MPSA_EINVAL, "mpsa_voigt: bad argument");
    if (n == 0) return MPSA_OK;
    MPSA_CUDA_TRY(cudaSetDevice(ctx->device));
    const int threads = 256;
    const int64_t blocks = (n + threads - 1) / threads;
    if (blocks > 0x7fffffff) return fail(MPSA_EINVAL, "mpsa_voigt: n = %lld too large", (long long)n);
    k_voigt_eval<<<(unsigned)blocks, threads, 0, (cudaStream_t)stream>>>(n, v, a, precision, out);
    MPSA_CUDA_TRY(cudaGetLastError());
    return MPSA_OK;
}

void mpsa_batch_destroy(mpsa_batch* b) {
    if (!b) return;
    cudaSetDevice(b->ctx->device);
    cudaDeviceSynchronize();
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    for (void* p : b->allocs) cudaFree(p);
    delete b;
}

}  // extern "C"
