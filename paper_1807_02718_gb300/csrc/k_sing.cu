// The 2D synthesis with the low-frequency split (Sec. 4.2; Sec. 5 steps
// T1b-T2d).
//
// Split synthesis.  For each window k and target x the inverse transform of
// F_k(w) = B_k^slow(w) V(x, w) over [-W, W] is, by F(-w) = conj F(w),
//   u_k(x, t) = (1/pi) Re[ I_{w_c}^{W}[F_k](t - s_k) + I_0^{w_c}[F_k](t - s_k) ]
// (eq. fourier_sing_decomp).  The smooth piece uses the n = J - j_c
// equispaced samples of [w_c, W] (w_c = omega_{j_c}): their FC(Gram)
// continuation (d = 6, C = 31, fc_gram_table.h) has period P = (n + C) dw, its
// DFT gives the coefficients of eq. fourier_approx about delta = (w_c + W)/2,
// and the term-wise integral eq. approx gives the transform at any t.  The
// singular piece uses the Filon-Clenshaw-Curtis rule on the graded mesh
// mu_j = w_c (j/4)^9.1 (eq. gradedmesh), 8 Clenshaw-Curtis points on each of
// the subintervals [mu_{j-1}, mu_j], j = 2..4 (eq. gradedmeshIntRule): the
// degree-7 interpolant times e^{-iwt} integrated exactly through the
// Chebyshev moments rho_n(kappa) = int_{-1}^{1} T_n(x) e^{-i kappa x} dx
// (power series, Gauss-Legendre for |kappa| < 12, the forward three-term
// recurrence above, where it is stable).
//
// Everything is linear in the frequency samples, so, as in the periodic
// synthesis, the target dependence is one real contraction:
//   u(x, t) = Re sum_p V'_p(x) G'_p(t),
// V' the target fields at the n smooth and 24 singular frequencies and
//   G'_p(t) = (1/pi) sum_k B_k(w_p) D_p(t - s_k),
// D_p the transform weight of sample p: for the smooth samples
// D_p(t') = sum_m K_m(t') E[m][p] with E = (shifted DFT) o (FC extension) and
// K_m(t') = e^{-i delta t'} 2A sinc((2A/P)(alpha t' - m)), alpha = P / (2 pi);
// for the singular samples the FCC weights.
//
// The L-term sums.  E is a shifted DFT after an extension that is the identity
// but for the 6 samples at either end, and with i = p - (n-1)/2, r = (n-1)/L
//   D_p = (2A/L) e^{-i delta t'} [S_i(y) + sum_j Xc[j][p] S_(n+j-(n-1)/2)(y)],
//   S_i(y) = sum_m sinc(r (y - m)) e^{-2 pi i m i / L},  y = alpha t',
// the sum over j (the continuation) for the end samples only, i modulo L.  S_i
// is the periodic synthesis's D_p with the kernel sinc(r .), band-limited to
// [-r pi, r pi] in y, and S_-i is its conjugate, so for i = 0..h (h = L/2):
//   |y| < 1.25 h: 42 samples of a table of S_i at the half-integers, built per
//     call (sinc_interp.cuh);
//   beyond: sin(pi r (y - m)) split into e^{+-i pi r (y - m)} and the Chebyshev
//     expansion of 1/(y - m) (k_synth.cu): with F_l(rho) = sum_q rho^q sum_m T_q(m/h)
//     e^{-2 pi i m l / L} (the far-field table of the periodic path, order L),
//     S_i = a F_(i+(n-1)/2) + conj(a) F_(i-(n-1)/2).
// Per (time, window) that is about 500 packed instructions for each of h + 1
// values in place of L of them for each of n.
#include <cmath>

#include "dfloat.cuh"
#include "fc_gram_table.h"
#include "fh_internal.h"
#include "scratch.cuh"
#include "sinc_interp.cuh"

namespace fh {
namespace {

constexpr int kSM = 4, kSNq = 8;
constexpr double kSQ = 9.1;
constexpr int kNsing = (kSM - 1) * kSNq;
constexpr int kGl = 24;    // Gauss-Legendre nodes, symmetric: the positive half is kept
constexpr int kMom = 13;   // terms of the moments' power series in kappa^2

// Constants of the rule: an argument of the launch (constant memory), so that calls
// with other meshes on other streams keep theirs.
struct FccRule {
    double cheb[kSNq][kSNq];   // interpolant coefficients a_n = sum_c cheb[n][c] f_c
    double glx[kGl / 2], glw[kGl / 2];
    double mom[kSNq][kMom];    // int T_n x^q dx / q!, q = 2 m + n mod 2
    double mu[kSM];            // graded mesh
};

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 expi(double th) {
    double s, c;
    sincos(th, &s, &c);
    return make_double2(c, s);
}
// Continuation rows: Xc[j * n + p] = d e_j / d f_p (right end blended to
// zero, plus the left end read backwards, blended and reversed); and the FP64
// phases ph[q] = e^{-2 pi i q / L}, q < L = n + kFcC.
__global__ void fc_rows_kernel(int n, double *__restrict__ Xc, double2 *__restrict__ ph) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (j == 0 && p < n + kFcC) {
        double sn, cs;
        sincospi(-2.0 * (double)p / (double)(n + kFcC), &sn, &cs);
        ph[p] = make_double2(cs, sn);
    }
    if (p >= n) return;
    double v = 0.0;
    if (p >= n - kFcD) {
        const int i = p - (n - kFcD);
        for (int k = 0; k < kFcD; ++k) v += kFcA[j][k] * kFcQ[i][k];
    }
    if (p < kFcD) {
        const int i = kFcD - 1 - p;
        for (int k = 0; k < kFcD; ++k) v += kFcA[kFcC - 1 - j][k] * kFcQ[i][k];
    }
    Xc[(long long)j * n + p] = v;
}

// sinc(r v / 2) for integers v, r = num / L: the phase pi num v / (2 L) is reduced in integers.
__device__ __forceinline__ double sinc_half(int num, int L, long long v) {
    if (v == 0) return 1.0;
    const long long k = (long long)num * v;
    return sinpi((double)(k % (4LL * L)) / (2.0 * L)) * (2.0 * L) / (kPi * (double)k);
}

constexpr int kMid = kFcC / 2;    // continuation point kMid has the frequency index h
constexpr int kTop = kMid + 1 + kFcD;        // S_(h - kTop + 1) .. S_h enter the end samples' weights

// Table of S_i(g/2), |g| <= G, i = 0..h: tab[(g + G) hp + i] = (re hi, im hi, re
// lo, im lo), hp = h + 1.  One CTA per kTabRows rows g >= 0 and 128 columns; m and
// -m are paired, their sinc sums staged in chunks of kTabChunk for all columns;
// the rows -g from S_i(-y) = conj S_i(y) + (-1)^i (sinc(r (y - h)) - sinc(r (y + h))).
// The CTAs of the first columns also form top[(g + G) kTop + q] = S_(h-q)(g/2),
// q < kTop, in FP64 (one thread per row and q).  0.13 ms for n = 251, 0.11 without.
constexpr int kTabRows = 4, kTabChunk = 256;

__global__ void __launch_bounds__(128) split_table_kernel(int num, int L, int G, const float4 *__restrict__ ph,
                                                          const double2 *__restrict__ ph64, float4 *__restrict__ tab,
                                                          double2 *__restrict__ top) {
    const int h = L / 2, hp = h + 1, i = blockIdx.y * 128 + threadIdx.x, g0 = kTabRows * blockIdx.x;
    __shared__ float4 sc[kTabRows][kTabChunk];   // sinc(r (y - m)) +- sinc(r (y + m))
    __shared__ double2 sd[kTabRows][kTabChunk];
    static_assert(kTabRows * kTop <= 128, "a thread per row and top column");
    const bool first = blockIdx.y == 0, fp64 = first && threadIdx.x < kTabRows * kTop;
    const int tq = fp64 ? threadIdx.x / kTop : 0, ti = h - (fp64 ? threadIdx.x % kTop : 0), tg = g0 + tq;
    double2 td = make_double2(0.0, 0.0);
    int tk = 0;
    if (fp64) td.x = sinc_half(num, L, tg) + ((ti & 1) ? -1.0 : 1.0) * sinc_half(num, L, tg + 2LL * h);
    float2 ah[kTabRows], al[kTabRows], ac[kTabRows];   // (re, im), compensated
#pragma unroll
    for (int q = 0; q < kTabRows; ++q) {
        const int g = g0 + q;
        const double e = sinc_half(num, L, g + 2LL * h);
        const dfv v = df_from(sinc_half(num, L, g) + ((i & 1) ? -e : e));
        ah[q] = p2(v.hi, 0.f);
        al[q] = p2(v.lo, 0.f);
        ac[q] = p2(0.f, 0.f);
    }
    int k = 0;   // m i mod L
    for (int m0 = 1; m0 < h; m0 += kTabChunk) {
        const int mc = min(kTabChunk, h - m0);
        __syncthreads();
        for (int e = threadIdx.x; e < kTabRows * mc; e += 128) {
            const int q = e / mc, m = m0 + e % mc;
            const double a = sinc_half(num, L, g0 + q - 2LL * m), b = sinc_half(num, L, g0 + q + 2LL * m);
            sc[q][e % mc] = df_pack(a + b, a - b);
            if (first) sd[q][e % mc] = make_double2(a + b, a - b);
        }
        __syncthreads();
        if (fp64)
#pragma unroll 4
            for (int m = 0; m < mc; ++m) {
                tk += ti;
                if (tk >= L) tk -= L;
                const double2 e = __ldg(ph64 + tk), v = sd[tq][m];
                td.x = fma(e.x, v.x, td.x);
                td.y = fma(e.y, v.y, td.y);
            }
        if (i < hp)
            for (int m = 0; m < mc; ++m) {
                k += i;
                if (k >= L) k -= L;
                const float4 e = __ldg(ph + k);   // e^{-2 pi i m i / L}
#pragma unroll
                for (int q = 0; q < kTabRows; ++q) {
                    const float4 v = sc[q][m];
                    df2_acc_c(ah[q], al[q], ac[q], {p2(e.x, e.z), p2(e.y, e.w)}, {p2(v.x, v.z), p2(v.y, v.w)});
                }
            }
    }
    if (fp64 && tg <= G) {
        double2 *row = top + threadIdx.x % kTop;
        row[(long long)(tg + G) * kTop] = td;
        const double c = sinc_half(num, L, tg - 2LL * h) - sinc_half(num, L, tg + 2LL * h);
        if (tg > 0) row[(long long)(G - tg) * kTop] = make_double2(td.x + ((ti & 1) ? -c : c), -td.y);
    }
    if (i >= hp) return;
#pragma unroll
    for (int q = 0; q < kTabRows; ++q) {
        const int g = g0 + q;
        if (g > G) break;
        const df2 t = df2_sum3(ah[q], al[q], ac[q]);
        tab[(long long)(g + G) * hp + i] = make_float4(t.h.x, t.h.y, t.l.x, t.l.y);
        const double c = sinc_half(num, L, g - 2LL * h) - sinc_half(num, L, g + 2LL * h);
        const dfv re = df_add(df2_x(t), df_from((i & 1) ? -c : c));
        if (g > 0) tab[(long long)(G - g) * hp + i] = make_float4(re.hi, -t.h.y, re.lo, -t.l.y);
    }
}

// sinc(2u) E(u) of sample row g0 + i in FP64 (as sinc_weight).
__device__ __forceinline__ double sinc_weight64(double uc, double s2, int gc, int g0, int i) {
    const double u = uc + 0.5 * (double)(gc - g0 - i);
    if (u == 0.0) return 1.0;
    const double x = u * u * (1.0 / (kSincU * kSincU));
    if (!(x < 1.0)) return 0.0;
    const double e = exp(-kSincBeta * x / (1.0 + sqrt(1.0 - x)));
    return (((g0 + i) & 1) ? -s2 : s2) * e / (2.0 * kPi * u);
}

// What a window contributes at one time (formed in FP64 by one thread).
struct SplitWindow {
    int R, R1;           // far terms and those taken in double-float; R = 0: near
    int g0, gc;          // near: first and nearest sample, y - gc/2 and sin(2 pi y)
    double uc, s2;
    dfv rho, ar, ai;     // far: ratio and the factor a
    double2 c;           // (2A/L) e^{-i delta t'} / pi, and in double-float
    dfv cr, ci;
};
constexpr int kSplitChunk = 32;   // windows whose constants are held at once
constexpr int kSplitThreads = 256;
constexpr int kEndPer = (kMid + 1) / 2;      // folded continuation terms per lane
constexpr int kTopParts = 4;      // interpolations of a top value side by side
static_assert(kFcC == 2 * kMid + 1 && 2 * kEndPer == kMid + 1, "continuation points in pairs about the middle one");
static_assert(4 * kFcD <= 32 && kTop <= 32, "one warp takes the end samples");
// The values a CTA keeps for its time: S_0 .. S_h, F_0 .. F_h and the sums of n samples.
constexpr int kSplitSmem = 200 * 1024;
constexpr int kSplitCtas = 4 * kSms;   // times per launch where they are in device memory
__host__ __device__ inline size_t split_work_bytes(int n) {
    const size_t hp = (size_t)(n + kFcC) / 2 + 1;
    return ((2 * hp + n) * sizeof(float4) + n * sizeof(float2) + 15) & ~(size_t)15;
}

// Smooth-piece weights: one CTA per time.  Per window S_0 .. S_h go to shared
// memory, then every interior sample adds B_k(w_p) D_p to its sum (shared memory,
// its thread's own; double-float with compensated low parts).
// The end samples: the continuation point j has index i = h - kMid + j modulo L, so
// that points kMid - q and kMid + q carry S_(h-q) and its conjugate, and sample n -
// kFcD + s (index h - kTop + 1 + s) has
//   Re D = Re S + Xc[kMid] Re S_h + sum_q (Xc[kMid - q] + Xc[kMid + q]) Re S_(h-q),
//   Im D = Im S + Xc[kMid] Im S_h + sum_q (Xc[kMid - q] - Xc[kMid + q]) Im S_(h-q),
// sample kFcD - 1 - s the conjugate.  The entries of Xc reach 6e4; they cancel for
// fields that are smooth from sample to sample, and for others every rounding
// before them shows in u.  So the S of near windows that enter here are FP64 (table,
// weights and sums), and the sums and products with B_k(w_p), one warp per window:
// 24 lanes (sample, part, half of the terms), then 12 lanes (end sample).
// Rows 0..n-1 of the weight planes: Gr = Re G / pi, Gm = -Im G / pi.
// kShared: the values of a time in shared memory (split_work_bytes(n) = 40 n + 528
// bytes, n <= 5106 at kSplitSmem); otherwise in `work`, the launch's CTAs taking
// the times from it0 on.
// Bound by the FP64 pipe (active 73 % of the cycles, the FMA pipe 36 %): splits of B for the
// interior samples, interpolation weights and constants per window, end samples.
// Measured (GB300; 1024 x 4096 samples, n = 251, 29 windows): 1.58 -> 0.99 ms, whole call
// 2.34 ms with 384 double-float products (end sample, continuation point) per window, each splitting
// its B in FP64, 1.74 ms so.  Error against extended precision over 28 meshes of
// n = 20..110: geometric mean 4.8e-12 -> 6.6e-13, largest 6.6e-11 -> 1.7e-11 (L-term
// double-float sums per sample: 2.0e-11 and 1.3e-10).
template <bool kShared>
__global__ void __launch_bounds__(kSplitThreads) smooth_weights_kernel(
    int it0, float4 *work, int n, int L, double A, double P, double delta, int K, const double *__restrict__ s,
    const double2 *__restrict__ B, int J, int j_c, const double *__restrict__ Xc, const float4 *__restrict__ tab,
    const double2 *__restrict__ top_tab, int G, const float4 *__restrict__ nu, const double *__restrict__ T, int n_T, double *__restrict__ Gr,
    double *__restrict__ Gm) {
    extern __shared__ float4 sm[];
    __shared__ SplitWindow win[kSplitChunk];
    __shared__ float2 swt[kSincPts];
    __shared__ double swd[kSincPts];
    __shared__ double2 tops[kTopParts][kTop];
    __shared__ double top[2][kTop];   // Re, Im S_(h-q)
    const int h = L / 2, hp = h + 1, nm = (n - 1) / 2, it = it0 + blockIdx.x, tid = threadIdx.x;
    float4 *Ss = kShared ? sm : work + blockIdx.x * (split_work_bytes(n) / sizeof(float4));
    float4 *Fs = Ss + hp, *acc = Ss + 2 * hp;   // S_i, F_l, G_p: (re hi, im hi, re lo, im lo)
    float2 *accc = reinterpret_cast<float2 *>(acc + n);   // G_p: third parts
    const double t = T[it];
    for (int p = tid; p < n; p += blockDim.x) {
        acc[p] = make_float4(0.f, 0.f, 0.f, 0.f);
        accc[p] = p2(0.f, 0.f);
    }
    // the last warp (it has the fewest interior samples): the folded
    // continuation terms of its lanes, and sums of end sample `lane`
    const bool ends = tid >= (int)blockDim.x - 32;
    const int lane = tid & 31, smp = min(lane >> 2, kFcD - 1), part = (lane >> 1) & 1, q0 = (lane & 1) * kEndPer;
    double xf[kEndPer];
    const int pe = lane < kFcD ? n - kFcD + lane : 2 * kFcD - 1 - min(lane, 2 * kFcD - 1);
    double2 ge = make_double2(0.0, 0.0);
    if (ends) {
        const double *x = Xc + n - kFcD + smp;
#pragma unroll
        for (int e = 0; e < kEndPer; ++e) {
            const int q = q0 + e;
            const double lo = x[(long long)(kMid - q) * n], hi = q ? x[(long long)(kMid + q) * n] : 0.0;
            xf[e] = part ? lo - hi : lo + hi;
        }
    }
    const double r = (double)(n - 1) / (double)L;
    for (int k0 = 0; k0 < K; k0 += kSplitChunk) {
        __syncthreads();
        for (int k = tid; k < min(kSplitChunk, K - k0); k += blockDim.x) {
            SplitWindow w;
            const double tp = t - s[k0 + k], y = P * tp * (0.5 / kPi), a = y / (double)h;
            w.R = w.R1 = 0;
            w.rho = w.ar = w.ai = df_make(0.f, 0.f);
            w.g0 = w.gc = 0;
            w.uc = w.s2 = 0.0;
            if (fabs(a) < 1.25) {
                w.gc = (int)rint(2.0 * y);
                w.g0 = (int)floor(2.0 * y) - (kSincPts / 2 - 1);
                w.uc = y - 0.5 * (double)w.gc;   // exact
                double sn, cs;
                sincospi(y, &sn, &cs);
                w.s2 = 2.0 * sn * cs;
            } else {
                const double sq = copysign(sqrt((a - 1.0) * (a + 1.0)), a);
                const double rho = 1.0 / (a + sq);
                // truncation from binary32 logarithms (a term count, not a value)
                const float lr = -logf(fabsf((float)rho));
                w.R = max(1, min((int)ceilf(48.f * 0.693147181f / lr), kFarTerms));
                w.R1 = max(1, min((int)ceilf((25.f * 0.693147181f + logf((float)w.R)) / lr), w.R));
                w.rho = df_from(rho);
                // a = e^{i pi r y} / (2 i) times 1/(pi r) and the expansion's factor 2/(h s)
                double sn, cs;
                sincospi(A * tp * (1.0 / kPi), &sn, &cs);   // r y = A t' / pi
                const double f = 1.0 / (kPi * r * (double)h * sq);
                w.ar = df_from(f * sn);
                w.ai = df_from(-f * cs);
            }
            const double2 ph = expi(-delta * tp);
            const double f = 2.0 * A / ((double)L * kPi);
            w.c = make_double2(f * ph.x, f * ph.y);
            w.cr = df_from(w.c.x);
            w.ci = df_from(w.c.y);
            win[k] = w;
        }
        for (int k = k0; k < min(k0 + kSplitChunk, K); ++k) {
            __syncthreads();   // the window constants; the previous window's S is used
            const SplitWindow &w = win[k - k0];
            if (w.R == 0) {
                if (tid < kSincPts) {
                    const double v64 = sinc_weight64(w.uc, w.s2, w.gc, w.g0, tid);
                    const dfv v = df_from(v64);
                    swt[tid] = p2(v.hi, v.lo);
                    swd[tid] = v64;
                }
                __syncthreads();
                const int te = (int)blockDim.x - 1 - tid;   // the top values: the last threads
                if (te < kTopParts * kTop) {
                    const int c = te / kTop, e = te % kTop;
                    const double2 *col = top_tab + (long long)(w.g0 + G) * kTop + e;
                    double2 v = make_double2(0.0, 0.0);
#pragma unroll 4
                    for (int q = c; q < kSincPts; q += kTopParts) {
                        const double2 x = __ldg(col + q * kTop);
                        v.x = fma(swd[q], x.x, v.x);
                        v.y = fma(swd[q], x.y, v.y);
                    }
                    tops[c][e] = v;
                }
                const float4 *row = tab + (long long)(w.g0 + G) * hp;
                for (int i = tid; i < hp - kTop; i += blockDim.x) {
                    float2 sh = p2(0.f, 0.f), sl = sh, sc = sh;
#pragma unroll 6
                    for (int q = 0; q < kSincPts; ++q) {
                        const float4 v = __ldg(row + (long long)q * hp + i);
                        const float2 wt = swt[q];
                        df2_acc_c(sh, sl, sc, {p2(wt.x, wt.x), p2(wt.y, wt.y)}, {p2(v.x, v.y), p2(v.z, v.w)});
                    }
                    const df2 v = df2_sum3(sh, sl, sc);
                    Ss[i] = make_float4(v.h.x, v.h.y, v.l.x, v.l.y);
                }
            } else {
                for (int l = tid; l < hp; l += blockDim.x) {   // F_(l + h)
                    float2 a = p2(0.f, 0.f);
                    const float2 rh = p2(w.rho.hi, w.rho.hi), rl = p2(w.rho.lo, w.rho.lo);
                    for (int q = w.R - 1; q >= w.R1; --q) {    // binary32 tail
                        const float4 v = __ldg(nu + (long long)q * hp + l);
                        a = p2_fma(a, rh, p2(v.x, v.y));
                    }
                    df2 f = {a, p2(0.f, 0.f)};
                    for (int q = w.R1 - 1; q >= 0; --q) {
                        const float4 v = __ldg(nu + (long long)q * hp + l);
                        float2 e;
                        const float2 p = p2_prod(f, {rh, rl}, e), c = p2(v.x, v.y), x = p2_add(p, c);
                        f = df2_quick(x, p2_add(p2_two_sum_err(p, c, x), p2_add(e, p2(v.z, v.w))));
                    }
                    Fs[l] = make_float4(f.h.x, f.h.y, f.l.x, f.l.y);
                }
                __syncthreads();
                const df2 ar = df2_bcast(w.ar), ai = df2_make(df_neg(w.ai), w.ai);
                for (int i = tid; i < hp; i += blockDim.x) {
                    auto F = [&](int l) {   // F_l, 0 <= l < L: F_(h - l) = conj F_(h + l)
                        const float4 v = Fs[l >= h ? l - h : h - l];
                        const float sg = l >= h ? 1.f : -1.f;
                        return df2{p2(v.x, sg * v.y), p2(v.z, sg * v.w)};
                    };
                    const df2 u = F(i + nm), v = F(i >= nm ? i - nm : i - nm + L);
                    // a u + conj(a) v = ar (u + v) + i ai (u - v)
                    const df2 sum = df2_add(u, v), dif = df2_add(u, {p2_neg(v.h), p2_neg(v.l)});
                    const df2 S = df2_dot2(ar, sum, ai, df2_swap(dif));
                    Ss[i] = make_float4(S.h.x, S.h.y, S.l.x, S.l.y);
                }
            }
            __syncthreads();
            auto S = [&](int i) {   // S_i, |i| <= h
                const float4 v = Ss[i < 0 ? -i : i];
                const float sg = i < 0 ? -1.f : 1.f;
                return df2{p2(v.x, sg * v.y), p2(v.z, sg * v.w)};
            };
            auto bc = [&](int p) {   // B_k(w_p) (2A/L) e^{-i delta t'} / pi
                const double2 b = B[(long long)k * J + j_c + p];
                const dfv br = df_from(b.x), bi = df_from(b.y);
                return df2_dot2(df2_bcast(br), df2_make(w.cr, w.ci), df2_make(df_neg(bi), bi), df2_make(w.ci, w.cr));
            };
            for (int p = kFcD + tid; p < n - kFcD; p += blockDim.x) {
                const df2 b = bc(p), x = S(p - nm), xs = df2_swap(x);
                const float4 q = acc[p];
                float2 gh = p2(q.x, q.y), gl = p2(q.z, q.w), gc = accc[p];
                df2_acc_c(gh, gl, gc, df2_bcast(df2_x(b)), x);
                df2_acc_c(gh, gl, gc, df2_make(df_neg(df2_y(b)), df2_y(b)), xs);
                acc[p] = make_float4(gh.x, gh.y, gl.x, gl.y);
                accc[p] = gc;
            }
            if (ends) {   // FP64
                if (lane < kTop) {
                    double2 v;
                    if (w.R == 0) {
                        v = tops[0][lane];
                        for (int c = 1; c < kTopParts; ++c) v = cadd(v, tops[c][lane]);
                    } else {
                        const float4 f = Ss[h - lane];
                        v = make_double2((double)f.x + (double)f.z, (double)f.y + (double)f.w);
                    }
                    top[0][lane] = v.x;
                    top[1][lane] = v.y;
                }
                const double2 b = B[(long long)k * J + j_c + pe], c = w.c;
                __syncwarp();
                double d = q0 ? 0.0 : top[part][kTop - 1 - smp];
#pragma unroll
                for (int e = 0; e < kEndPer; ++e) d = fma(xf[e], top[part][q0 + e], d);
                d += __shfl_xor_sync(0xffffffffu, d, 1);
                const int src = 4 * (lane < kFcD ? lane : min(lane, 2 * kFcD - 1) - kFcD);
                const double dr = __shfl_sync(0xffffffffu, d, src), di = __shfl_sync(0xffffffffu, d, src + 2);
                const double2 bw = cmul(b, c), v = cmul(bw, make_double2(dr, lane < kFcD ? di : -di));
                ge.x += v.x;
                ge.y += v.y;
            }
        }
    }
    __syncthreads();
    for (int p = kFcD + tid; p < n - kFcD; p += blockDim.x) {
        const float4 q = acc[p];
        const float2 c = accc[p];
        Gr[(long long)p * n_T + it] = (double)q.x + (double)q.z + (double)c.x;
        Gm[(long long)p * n_T + it] = -((double)q.y + (double)q.w + (double)c.y);
    }
    if (ends && lane < 2 * kFcD) {
        Gr[(long long)pe * n_T + it] = ge.x;
        Gm[(long long)pe * n_T + it] = -ge.y;
    }
}

// Chebyshev moments rho_n(kappa) = int_{-1}^{1} T_n(x) e^{-i kappa x} dx, n < 8: real
// for even n, imaginary for odd n (rho[n] holds the real or imaginary part).
//   |kappa| <= 2: their power series (mom[n][s] (-1)^s kappa^(2s), times -kappa
//     for odd n; the remainder is below 3e-17);
//   |kappa| < 12: 24-point Gauss-Legendre, x and -x together (error below 1e-17);
//   beyond: the forward three-term recurrence, stable there.
__device__ __forceinline__ void cheb_moments(const FccRule &rule, double kap, double (&rho)[kSNq]) {
    const double ka = fabs(kap);
    if (ka <= 2.0) {
        const double z = -kap * kap;
#pragma unroll
        for (int q = 0; q < kSNq; ++q) {
            double v = rule.mom[q][kMom - 1];
#pragma unroll
            for (int m = kMom - 2; m >= 0; --m) v = fma(v, z, rule.mom[q][m]);
            rho[q] = (q & 1) ? -kap * v : v;
        }
        return;
    }
    if (ka < 12.0) {
#pragma unroll
        for (int q = 0; q < kSNq; ++q) rho[q] = 0.0;
        for (int g = 0; g < kGl / 2; ++g) {
            const double x = rule.glx[g], x2 = 2.0 * x;
            double s, c;
            sincos(kap * x, &s, &c);
            c *= rule.glw[g];
            s *= -rule.glw[g];
            double t0 = 1.0, t1 = x;
#pragma unroll
            for (int q = 0; q < kSNq; ++q) {   // T_q(x) times the even (cos) or odd (-sin) part
                rho[q] = fma(t0, (q & 1) ? s : c, rho[q]);
                const double t2 = fma(x2, t1, -t0);
                t0 = t1;
                t1 = t2;
            }
        }
        return;
    }
    double sn, cs;
    sincos(kap, &sn, &cs);
    const double ik = 1.0 / kap;
    rho[0] = 2.0 * sn * ik;
    rho[1] = -2.0 * (sn - kap * cs) * ik * ik;
    const double x2 = 2.0 * ((kap * kap - 2.0) * sn + 2.0 * kap * cs) * ik * ik * ik;
    rho[2] = 2.0 * x2 - rho[0];
    // rho_{q+1} = (q+1)/(i kappa) [2 rho_q - (1/(q+1) - 1/(q-1)) sigma] + (q+1)/(q-1) rho_{q-1}, sigma =
    // e^{-i kappa} - (-1)^(q+1) e^{i kappa} = -2 i sin kappa (q odd) or 2 cos kappa (q even)
#pragma unroll
    for (int q = 2; q + 1 < kSNq; ++q) {
        const double f = 1.0 / (q + 1) - 1.0 / (q - 1), a = (double)(q + 1) * ik, e = (double)(q + 1) / (q - 1);
        // even q: rho_q real, bracket real b -> -i a b; odd q: bracket i b -> a b
        rho[q + 1] = (q & 1) ? fma(a, 2.0 * rho[q] + 2.0 * f * sn, e * rho[q - 1])
                             : fma(-a, 2.0 * rho[q] - 2.0 * f * cs, e * rho[q - 1]);
    }
}

// Singular-piece weights: one thread per (time, interval of the graded mesh,
// every kFccGroups-th window); the interval's eight Clenshaw-Curtis points
// share its Chebyshev moments and phase, computed once per window, and the
// window groups' sums are added in order.  Rows n .. n+23 of the weight planes
// (row n + 8 (jv - 1) + c for point c of interval jv).  Bound by the FP64 pipe:
// the moments took 32 sincos for |kappa| < 12 before
// (1.94 -> 0.34 ms at 4096 times, 29 windows).
constexpr int kFccTimes = 32, kFccGroups = 4;

__global__ void __launch_bounds__(kFccTimes *kFccGroups) fcc_weights_kernel(
    const __grid_constant__ FccRule rule, int n, int K, const double *__restrict__ s, const double2 *__restrict__ Bs,
    const double *__restrict__ T, int n_T, double *__restrict__ Gr, double *__restrict__ Gm) {
    __shared__ double2 sums[kFccGroups][kSNq][kFccTimes];
    const int lane = threadIdx.x % kFccTimes, grp = threadIdx.x / kFccTimes;
    const int it = blockIdx.x * kFccTimes + lane, jv = blockIdx.y + 1;
    const double a = rule.mu[jv - 1], b = rule.mu[jv];        // interval [mu_{jv-1}, mu_jv] (0-based)
    const double h = 0.5 * (b - a), dl = 0.5 * (a + b);
    const int i0 = (jv - 1) * kSNq;
    double2 acc[kSNq];
#pragma unroll
    for (int c = 0; c < kSNq; ++c) acc[c] = make_double2(0.0, 0.0);
    if (it < n_T) {
        const double t = T[it];
        for (int k = grp; k < K; k += kFccGroups) {
            const double tp = t - s[k];
            double rho[kSNq];
            cheb_moments(rule, h * tp, rho);
            double2 ph = expi(-dl * tp);
            ph.x *= h;
            ph.y *= h;
#pragma unroll
            for (int c = 0; c < kSNq; ++c) {
                double2 w = make_double2(0.0, 0.0);
#pragma unroll
                for (int q = 0; q < kSNq; q += 2) {
                    w.x = fma(rule.cheb[q][c], rho[q], w.x);
                    w.y = fma(rule.cheb[q + 1][c], rho[q + 1], w.y);
                }
                w = cmul(w, ph);
                const double2 bb = Bs[(long long)k * kNsing + i0 + c];
                acc[c].x = fma(bb.x, w.x, fma(-bb.y, w.y, acc[c].x));
                acc[c].y = fma(bb.x, w.y, fma(bb.y, w.x, acc[c].y));
            }
        }
    }
#pragma unroll
    for (int c = 0; c < kSNq; ++c) sums[grp][c][lane] = acc[c];
    __syncthreads();
    for (int e = threadIdx.x; e < kSNq * kFccTimes; e += kFccTimes * kFccGroups) {
        const int c = e / kFccTimes, l = e % kFccTimes, ti = blockIdx.x * kFccTimes + l;
        if (ti >= n_T) continue;
        double2 v = sums[0][c][l];
        for (int g = 1; g < kFccGroups; ++g) v = cadd(v, sums[g][c][l]);
        Gr[(long long)(n + i0 + c) * n_T + ti] = v.x / kPi;
        Gm[(long long)(n + i0 + c) * n_T + ti] = -v.y / kPi;
    }
}

// V' = [V rows j_c .. J-1 ; Vs rows 0 .. 23]
__global__ void stack_fields_kernel(int n, int n_x, int j_c, const double2 *__restrict__ V,
                                    const double2 *__restrict__ Vs, double2 *__restrict__ Vp) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, p = blockIdx.y;
    if (x >= n_x) return;
    Vp[(long long)p * n_x + x] = p < n ? V[(long long)(j_c + p) * n_x + x] : Vs[(long long)(p - n) * n_x + x];
}

// ---- host helpers ----

unsigned grid_of(long long n, int block) { return (unsigned)((n + block - 1) / block); }

// Gauss-Legendre nodes and weights on [-1, 1] (Newton's method on P_n).
void gauss_legendre(int n, double *x, double *w) {
    for (int i = 0; i < n; ++i) {
        double z = std::cos(kPi * (i + 0.75) / (n + 0.5)), dp = 0.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = z;
            for (int k = 2; k <= n; ++k) {
                const double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            dp = n * (z * p1 - p0) / (z * z - 1.0);
            const double dz = p1 / dp;
            z -= dz;
            if (std::fabs(dz) < 1e-16) break;
        }
        x[i] = z;
        w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
}

// mom[n][m] = int_{-1}^{1} T_n(x) x^q dx / q! with q = 2 m + n mod 2 (extended
// precision: the monomial terms of T_7 cancel by two digits).
void cheb_power_moments(double (&mom)[kSNq][kMom]) {
    long double c[kSNq][kSNq] = {};   // T_n = sum_k c[n][k] x^k
    c[0][0] = c[1][1] = 1.0L;
    for (int n = 2; n < kSNq; ++n)
        for (int k = 0; k < kSNq; ++k) c[n][k] = (k ? 2.0L * c[n - 1][k - 1] : 0.0L) - c[n - 2][k];
    for (int n = 0; n < kSNq; ++n)
        for (int m = 0; m < kMom; ++m) {
            const int q = 2 * m + (n & 1);
            long double v = 0.0L, f = 1.0L;
            for (int k = 0; k <= n; ++k)
                if (!((k + q) & 1)) v += c[n][k] * 2.0L / (k + q + 1);
            for (int k = 2; k <= q; ++k) f *= k;
            mom[n][m] = (double)(v / f);
        }
}

}  // namespace
}  // namespace fh

using namespace fh;

extern "C" fh_status fh_sing_frequencies(double omega_c, double *out) {
    if (!out || !(omega_c > 0.0) || !std::isfinite(omega_c)) return FH_EINVAL;
    for (int jv = 1; jv < kSM; ++jv) {
        const double a = omega_c * std::pow((double)jv / kSM, kSQ);
        const double b = omega_c * std::pow((double)(jv + 1) / kSM, kSQ);
        for (int c = 0; c < kSNq; ++c)
            out[(jv - 1) * kSNq + c] = 0.5 * (a + b) + 0.5 * (b - a) * std::cos(kPi * c / (kSNq - 1));
    }
    return FH_OK;
}

extern "C" fh_status fh_synthesize_sing(int J, double W, int j_c, int K, const double *d_s, const double *d_B,
                                        const double *d_Bs, const double *d_V, const double *d_Vs, int n_x,
                                        const double *d_T, int n_T, double *d_u, void *stream) {
    if (J < 2 || !(W > 0.0) || K < 1 || n_x < 0 || n_T < 0 || j_c < 1) return FH_EINVAL;
    const int n = J - j_c;
    if (n < 2 * kFcD || ((n + kFcC) & 1)) return FH_EINVAL;   // FC needs 2d samples; n + C even
    if (n + kNsing > 65535) return FH_EINVAL;                  // rows of the stacked fields are in grid.y
    if (n_x == 0 || n_T == 0) return FH_OK;
    if (!d_s || !d_B || !d_Bs || !d_V || !d_Vs || !d_T || !d_u) return FH_EINVAL;
    if (cudaPeekAtLastError() != cudaSuccess) return FH_ECUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const double dw = W / (J - 1), wc = j_c * dw;
    const int L = n + kFcC, ns = n + kNsing;
    FccRule rule;
    double glx[kGl], glw[kGl];
    for (int q = 0; q < kSNq; ++q)
        for (int c = 0; c < kSNq; ++c) {
            const double wt = (c == 0 || c == kSNq - 1) ? 0.5 : 1.0;
            double v = 2.0 / (kSNq - 1) * wt * std::cos(kPi * q * c / (kSNq - 1));
            if (q == 0 || q == kSNq - 1) v *= 0.5;
            rule.cheb[q][c] = v;
        }
    gauss_legendre(kGl, glx, glw);
    for (int g = 0; g < kGl / 2; ++g) {   // node x and -x (the first half is positive)
        rule.glx[g] = glx[g];
        rule.glw[g] = 2.0 * glw[g];
    }
    cheb_power_moments(rule.mom);
    for (int j = 0; j < kSM; ++j) rule.mu[j] = wc * std::pow((double)(j + 1) / kSM, kSQ);
    fh_status status = FH_OK;
    {
        Scratch sc{{}, st};
        // half-integer table of S_i, far-field table of order L with its phases and powers
        const int h = L / 2, hp = h + 1, G = (5 * h + 1) / 2 + 24;
        float4 *tab = sc.get<float4>((size_t)(2 * G + 1) * hp);
        double2 *top = sc.get<double2>((size_t)(2 * G + 1) * kTop + L + ((size_t)kFcC * n + 1) / 2);
        double2 *ph64 = top + (size_t)(2 * G + 1) * kTop;             // and the continuation rows, one allocation
        double *Xc = reinterpret_cast<double *>(ph64 + L);
        float4 *nu = sc.get<float4>((size_t)kFarTerms * hp);
        float4 *ph = sc.get<float4>((size_t)L);
        double *pw = sc.get<double>((size_t)L * kFarTerms);
        double2 *Vp = sc.get<double2>((size_t)ns * n_x);
        double *Gr = sc.get<double>((size_t)ns * n_T);
        double *Gm = sc.get<double>((size_t)ns * n_T);
        const size_t work_bytes = split_work_bytes(n);
        const bool in_memory = work_bytes > kSplitSmem;
        float4 *work = in_memory ? sc.get<float4>(work_bytes / sizeof(float4) * std::min(kSplitCtas, n_T)) : nullptr;
        if ((in_memory && !work) || !tab || !top || !nu || !ph || !pw || !Vp || !Gr || !Gm) {
            cudaGetLastError();
            return FH_ENOMEM;
        }
        fc_rows_kernel<<<dim3(grid_of(L, 128), kFcC), 128, 0, st>>>(n, Xc, ph64);
        launch_far_table(hp, L, pw, nullptr, nu, ph, st);
        split_table_kernel<<<dim3(G / kTabRows + 1, grid_of(hp, 128)), 128, 0, st>>>(n - 1, L, G, ph, ph64, tab, top);
        const double A = 0.5 * (W - wc), P = L * dw, delta = 0.5 * (wc + W);
        // as many threads as values S_i (the longest loops), at least 128 for the end samples
        const int threads = std::min(kSplitThreads, std::max(128, (hp + 31) / 32 * 32));
        if (!work) {
            static std::atomic<unsigned long long> attr{0};
            ensure_smem_attr((const void *)smooth_weights_kernel<true>, kSplitSmem, attr);
            smooth_weights_kernel<true><<<n_T, threads, work_bytes, st>>>(
                0, nullptr, n, L, A, P, delta, K, d_s, reinterpret_cast<const double2 *>(d_B), J, j_c, Xc, tab, top, G,
                nu, d_T, n_T, Gr, Gm);
        } else {
            for (int it0 = 0; it0 < n_T; it0 += kSplitCtas)
                smooth_weights_kernel<false><<<std::min(kSplitCtas, n_T - it0), threads, 0, st>>>(
                    it0, work, n, L, A, P, delta, K, d_s, reinterpret_cast<const double2 *>(d_B), J, j_c, Xc, tab, top,
                    G, nu, d_T, n_T, Gr, Gm);
        }
        fcc_weights_kernel<<<dim3(grid_of(n_T, kFccTimes), kSM - 1), kFccTimes * kFccGroups, 0, st>>>(
            rule, n, K, d_s, reinterpret_cast<const double2 *>(d_Bs), d_T, n_T, Gr, Gm);
        stack_fields_kernel<<<dim3(grid_of(n_x, 128), ns), 128, 0, st>>>(
            n, n_x, j_c, reinterpret_cast<const double2 *>(d_V), reinterpret_cast<const double2 *>(d_Vs), Vp);
        unsigned char *slices = contract_slices_fp64(ns, n_x, n_T)
                                    ? sc.get<unsigned char>(contract_tc_scratch_bytes(ns, n_x, n_T)) : nullptr;
        if (slices) {
            if (launch_contract_tc(ns, n_x, n_T, Vp, Gr, Gm, d_u, slices, nullptr, st) != cudaSuccess) status = FH_ECUDA;
        } else {
            if (cudaPeekAtLastError() == cudaErrorMemoryAllocation) cudaGetLastError();   // no room for the slices
            launch_synth_contract(ns, n_x, n_T, Vp, Gr, Gm, d_u, st);
        }
        if (cudaGetLastError() != cudaSuccess) status = FH_ECUDA;
    }
    return status;
}
