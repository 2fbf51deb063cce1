// Steps a6-a7 (steps T0-T6): band-limited recentred synthesis of u(x, t).
//
// The paper expands F(omega) = B_k^slow(omega) V(x, omega) on [-W, W) in a
// trigonometric series from its values at M = 2(J-1) equispaced nodes (Sec.
// 4.1 eq. fourier_approx, P = 2W) and integrates it exactly against
// e^{-i omega (t - s_k)} (eq. approx), giving per window
//   u_k(x, t) = Re[(1/2pi) sum_m c_m 2W sinc(W (t - s_k)/pi - m)],
// summed over k (step T5, eq. uk_def).  Exchanging the (linear) sums yields
// the same numbers as a contraction over the non-negative frequencies p:
//   u(x, t) = sum_p Re[V(x, w_p) G_p(t)],
//   G_p(t)  = (mu_p / 2pi) sum_k B_k^slow(w_p) D_p(t - s_k),
//   D_p(tau) = (2W/M) sum_{m=-h}^{h-1} e^{-2 pi i m p / M} sinc(W tau/pi - m),
// with h = M/2, mu_0 = mu_{J-1} = 1 and mu_p = 2 otherwise (the nodes -w_p
// carry conj F since the signal is real).  The weights G are independent of
// the targets (the O(1)-in-T part); the contraction over p is a real GEMM
// u = [Vr | Vi] [Gr ; -Gi] with inner dimension 2J.
//
// D_p for windows far from t (|y| >= 1.25 h, y = W tau/pi) uses the Chebyshev
// expansion of 1/(y - m) in x = m/h on [-1, 1]: with a = y/h,
// s = sign(a) sqrt(a^2 - 1) and rho = 1/(a + s) (|rho| <= 1/2 for |a| >= 1.25),
//   1/(a - x) = (2/s) [1/2 + sum_{r>=1} rho^r T_r(x)]
// (the generating function of the Chebyshev polynomials), so that
//   D_p = (2W/M) (sin(pi y)/pi) (2/(h s)) sum_r rho^r nu_{p,r},
//   nu_{p,r} = sum_m (-1)^m T_r(m/h) e^{-2 pi i m p / M}  (r = 0 halved),
// truncated once |rho|^r < 2^-48 (|nu_{p,r}| <= M) and summed by Horner's
// rule in double-float arithmetic, except the terms past R1 with
// |rho|^R1 <= 2^-25 / R, which Horner's rule takes in FP32 first (their
// relative error ~R 2^-24 enters scaled by |rho|^R1, the size of the
// truncation error).  Its ratio |rho| is below the Taylor ratio h/|y| (0.5
// against 0.8 at |y| = 1.25 h), hence fewer terms.  Near windows interpolate a
// table of the direct sums or sum the M terms directly.
#include "dfloat.cuh"
#include "fh_internal.h"
#include "sinc_interp.cuh"

namespace fh {
namespace {

// nu_{p,r} as a contraction: pw[m + h][r] = T_r(m/h) (three-term recurrence
// T_{r+1} = 2x T_r - T_{r-1}, stable on [-1, 1]; T_0 halved; one thread per
// m), then one CTA per p stages (-1)^k (cos, sin)(2 pi k p / M) of a chunk of
// k in shared memory and thread r accumulates the cosine (even r) or sine
// (odd r) sum over k = 1 .. h-1, m and -m paired.
__global__ void far_powers_kernel(int M, double *__restrict__ pw) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= M) return;
    const int h = M / 2;
    const double xv = (double)(q - h) / (double)h;
    double t0 = 1.0, t1 = xv;
    pw[(long long)q * kFarTerms] = 0.5;
    for (int r = 1; r < kFarTerms; ++r) {
        pw[(long long)q * kFarTerms + r] = t1;
        const double t2 = 2.0 * xv * t1 - t0;
        t0 = t1;
        t1 = t2;
    }
}

constexpr int kFarChunk = 128;

__global__ void __launch_bounds__(128) far_table_kernel(int J, int M, const double *__restrict__ pw,
                                                       double2 *__restrict__ nu, float4 *__restrict__ nu_f,
                                                       float4 *__restrict__ ph) {
    const int p = blockIdx.x;
    const int r = threadIdx.x;
    const int h = M / 2;
    __shared__ double2 phs[kFarChunk];
    if (p == 0)
        for (int q = r; q < M; q += blockDim.x) {
            double sn, cs;
            sincospi(-2.0 * (double)q / (double)M, &sn, &cs);
            const float ch = (float)cs, sh = (float)sn;   // double-float (cos, sin)
            ph[q] = make_float4(ch, (float)(cs - (double)ch), sh, (float)(sn - (double)sh));
        }
    // Pairing m with -m (T_r(-x) = (-1)^r T_r(x), e^{-i th m} + (-1)^r e^{i th m} =
    // 2 cos(th m) for even r, -2i sin(th m) for odd r; th = 2 pi p / M):
    //   nu_{p,r} = T_r(0) + (-1)^(h+p+r) T_r(1)
    //            + 2 sum_{k=1}^{h-1} (-1)^k T_r(k/h) {cos(th k) | -i sin(th k)},
    // the m = -h term using e^{i th h} = (-1)^p (T_0 halved throughout).
    const bool odd_r = r & 1;
    double acc = 0.0;
    for (int k0 = 1; k0 < h; k0 += kFarChunk) {
        __syncthreads();
        for (int e = r; e < kFarChunk; e += blockDim.x) {
            const int k = k0 + e;
            double2 v = make_double2(0.0, 0.0);
            if (k < h) {
                const int q = (int)(((long long)k * p) % M);
                double sn, cs;
                sincospi(2.0 * (double)q / (double)M, &sn, &cs);
                const double sg = (k & 1) ? -1.0 : 1.0;
                v = make_double2(sg * cs, sg * sn);
            }
            phs[e] = v;
        }
        __syncthreads();
        if (r < kFarTerms) {
            const int ke = min(kFarChunk, h - k0);
            const double *col = pw + (long long)(k0 + h) * kFarTerms + r;
            for (int e = 0; e < ke; ++e) {
                const double w = col[(long long)e * kFarTerms];
                acc = fma(w, odd_r ? phs[e].y : phs[e].x, acc);
            }
        }
    }
    double sr = 0.0, si = 0.0;
    if (r < kFarTerms) {
        const double t0 = pw[(long long)h * kFarTerms + r];      // T_r(0) (T_0 halved)
        const double t1 = r == 0 ? 0.5 : 1.0;                    // T_r(1)
        const double edge = ((h + p + r) & 1) ? -t1 : t1;        // the m = -h term
        sr = t0 + edge + (odd_r ? 0.0 : 2.0 * acc);
        si = odd_r ? -2.0 * acc : 0.0;
    }
    if (r < kFarTerms) {
        if (nu) nu[(long long)r * J + p] = make_double2(sr, si);
        const float rh = (float)sr, ih = (float)si;   // double-float copy for the far Horner
        nu_f[(long long)r * J + p] = make_float4(rh, ih, (float)(sr - (double)rh), (float)(si - (double)ih));
    }
}

// Double-float (FP32 pair) arithmetic for the near-window sums: FP32 runs at
// 64x the FP64 rate on this GPU.  A value is hi + lo with |lo| <= ulp(hi)/2;
// products use the exact FMA residual (Dekker / Ogita-Rump-Oishi two-product),
// sums the two-sum of Knuth, giving ~2^-44 relative accuracy per operation.
struct dfl { float hi, lo; };

__device__ __forceinline__ dfl df_split(double v) {
    const float h = (float)v;
    return {h, (float)(v - (double)h)};
}

// acc += a * b (a, b double-float; acc double-float)
__device__ __forceinline__ void df_mac(float &sh, float &sl, dfl a, dfl b) {
    const float p = a.hi * b.hi;
    float pe = fmaf(a.hi, b.hi, -p);
    pe = fmaf(a.hi, b.lo, pe);
    pe = fmaf(a.lo, b.hi, pe);
    const float t = sh + p;
    const float z = t - sh;
    const float err = (sh - (t - z)) + (p - z);
    sl += err + pe;
    sh = t;
}

// a * b in double-float, renormalised
__device__ __forceinline__ dfl df_mulq(dfl a, dfl b) {
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    const float h = p + e;
    return {h, e - (h - p)};
}

// a + b and 1 / a in double-float, renormalised
__device__ __forceinline__ dfl df_addq(dfl a, dfl b) {
    const float sum = a.hi + b.hi;
    const float bb = sum - a.hi;
    const float e = ((a.hi - (sum - bb)) + (b.hi - bb)) + (a.lo + b.lo);
    const float h = sum + e;
    return {h, e - (h - sum)};
}

__device__ __forceinline__ dfl df_rcpq(dfl a) {
    const float r = 1.0f / a.hi;
    const float t = fmaf(-a.hi, r, 1.0f) - a.lo * r;
    const float h = r + r * t;
    return {h, r * t - (h - r)};
}

// a * r + v in double-float (r, v double-float; a updated)
__device__ __forceinline__ void df_horner(float &ah, float &al, dfl r, float vh, float vl) {
    const float p = ah * r.hi;
    float e = fmaf(ah, r.hi, -p);
    e = fmaf(ah, r.lo, e);
    e = fmaf(al, r.hi, e);
    const float s = p + vh;
    const float bb = s - p;
    float err = (p - (s - bb)) + (vh - bb);
    err += e + vl;
    ah = s + err;
    al = err - (ah - s);
}

__device__ __forceinline__ dfl df_negq(dfl a) { return {-a.hi, -a.lo}; }

// Direct near-window sum, unscaled, for the thread's p (all threads of the CTA
// call it; it begins and ends with a barrier):
//   (rh + rl) + i (ih + il) = sum_{m=-h}^{h-1} e^{-2 pi i m p / M} sinc(y - m)
//   = S(y) + (-1)^p S(y+h) + sum_{j=1}^{h-1} (cos_j (S(y-j) + S(y+j))
//     + i sin_j (S(y-j) - S(y+j))),
// S(v) = sinc(v), (cos_j, sin_j) the phase e^{-2 pi i j p / M} (its conjugate
// pairs -j with j).  The sinc row uses sin(pi (y - j)) = (-1)^j sin(pi y);
// sypi = sin(pi y) / pi.  ph4: M phases (shared), sc4: h + 1 float4 (shared).
__device__ void stage_sinc_row(double y, dfl sypi, int h, float4 *sc4) {
    for (int jj = threadIdx.x; jj < h + 1; jj += blockDim.x) {
        // jj = 0: S(y) and S(y + h) into slot 0; jj >= 1: S(y - jj) +- S(y + jj)
        const int ja = jj == 0 ? 0 : jj, jb = jj == 0 ? h : jj;
        dfl va, vb;
        {
            const double d = y - (double)ja;
            if (d == 0.0) va = {1.f, 0.f};
            else {
                va = df_mulq(sypi, df_rcpq(df_split(d)));
                if (ja & 1) va = {-va.hi, -va.lo};
            }
        }
        {
            const double d = y + (double)jb;
            if (d == 0.0) vb = {1.f, 0.f};
            else {
                vb = df_mulq(sypi, df_rcpq(df_split(d)));
                if (jb & 1) vb = {-vb.hi, -vb.lo};
            }
        }
        if (jj == 0) {
            sc4[0] = make_float4(va.hi, va.lo, vb.hi, vb.lo);   // S(y), S(y + h)
        } else if (jj < h) {
            const dfl sp = df_addq(va, vb), sm = df_addq(va, {-vb.hi, -vb.lo});
            sc4[jj] = make_float4(sp.hi, sp.lo, sm.hi, sm.lo);
        }
    }
}

__device__ void near_sum(double y, dfl sypi, int h, int M, int p, int J, const float4 *ph4,
                         float4 *sc4, float &rh, float &rl, float &ih, float &il) {
    __syncthreads();
    stage_sinc_row(y, sypi, h, sc4);
    __syncthreads();
    rh = rl = ih = il = 0.f;
    if (p < J) {
        const float4 s0 = sc4[0];
        const dfl r0 = df_addq({s0.x, s0.y}, (p & 1) ? dfl{-s0.z, -s0.w} : dfl{s0.z, s0.w});
        rh = r0.hi;
        rl = r0.lo;
        int q = p;
        for (int jj = 1; jj < h; ++jj) {
            const float4 e = ph4[q];     // one 16-byte gather: cos and sin
            const float4 v = sc4[jj];    // one 16-byte broadcast: both sinc sums
            df_mac(rh, rl, {e.x, e.y}, {v.x, v.y});
            df_mac(ih, il, {e.z, e.w}, {v.z, v.w});
            q += p;
            if (q >= M) q -= M;
            if ((jj & 31) == 31) {   // renormalise the accumulators
                float tr = rh + rl; rl = rl - (tr - rh); rh = tr;
                float ti = ih + il; il = il - (ti - ih); ih = ti;
            }
        }
    }
}

// The sampled near sums.  Odd rows (direct sums, sin(pi g / 2) = +-1): one
// CTA per kTabRows consecutive positive odd rows and kTabThreads columns p,
// so that each phase gathered from shared memory serves kTabRows rows; the
// negative odd rows follow from the positive ones by a conjugation and a
// real end-term correction.  Even rows:
// D_p(n) = e^{-2 pi i n p / M} for -h <= n < h, else 0 (sinc(n - m) vanishes
// off m = n), written by the CTAs past the odd ones (grid-stride, blockIdx.y
// 0 only).
constexpr int kTabRows = 4;
constexpr int kTabThreads = 128;

__global__ void __launch_bounds__(kTabThreads) sinc_table_kernel(int J, int M, int G, int odd_ctas,
                                                                 const float4 *__restrict__ ph_g,
                                                                 float4 *__restrict__ tab) {
    const int h = M / 2;
    if ((int)blockIdx.x >= odd_ctas) {
        if (blockIdx.y != 0) return;
        const int e_first = (G & 1) ? 1 - G : -G;           // first even row
        const long long n_even = (long long)((G - e_first) / 2 + 1) * J;
        const int nb = gridDim.x - odd_ctas;
        for (long long idx = (long long)(blockIdx.x - odd_ctas) * blockDim.x + threadIdx.x; idx < n_even;
             idx += (long long)nb * blockDim.x) {
            const int pp = (int)(idx % J);
            const int g = e_first + 2 * (int)(idx / J);
            const int n = g / 2;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (n >= -h && n < h) {
                const float4 e = ph_g[(long long)(n + M) * pp % M];
                v = make_float4(e.x, e.z, e.y, e.w);
            }
            tab[(long long)(g + G) * J + pp] = v;
        }
        return;
    }
    extern __shared__ __align__(16) float4 sm4[];
    float4 *ph4 = sm4;        // M phases
    float4 *sc4 = sm4 + M;    // kTabRows rows of h sinc sums
    const int g0 = 1 + 2 * kTabRows * (int)blockIdx.x;   // positive odd rows; -g from g
    const int p = blockIdx.y * kTabThreads + threadIdx.x;
    for (int q = threadIdx.x; q < M; q += blockDim.x) ph4[q] = ph_g[q];
#pragma unroll 1
    for (int r = 0; r < kTabRows; ++r) {
        const int g = g0 + 2 * r;
        if (g <= G) {
            const double sy = (g & 3) == 1 ? 1.0 : -1.0;   // sin(pi g / 2)
            stage_sinc_row(0.5 * (double)g, df_split(sy / kPi), h, sc4 + r * h);
        } else {
            for (int jj = threadIdx.x; jj < h; jj += blockDim.x) sc4[r * h + jj] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    __syncthreads();
    if (p >= J) return;
    float ac[kTabRows][4];
#pragma unroll
    for (int r = 0; r < kTabRows; ++r) {
        const float4 s0 = sc4[r * h];
        const dfl r0 = df_addq({s0.x, s0.y}, (p & 1) ? dfl{-s0.z, -s0.w} : dfl{s0.z, s0.w});
        ac[r][0] = r0.hi;
        ac[r][1] = r0.lo;
        ac[r][2] = ac[r][3] = 0.f;
    }
    int q = p;
    for (int jj = 1; jj < h; ++jj) {
        const float4 e = ph4[q];
#pragma unroll
        for (int r = 0; r < kTabRows; ++r) {
            const float4 v = sc4[r * h + jj];
            df_mac(ac[r][0], ac[r][1], {e.x, e.y}, {v.x, v.y});
            df_mac(ac[r][2], ac[r][3], {e.z, e.w}, {v.z, v.w});
        }
        q += p;
        if (q >= M) q -= M;
        if ((jj & 31) == 31) {   // renormalise the accumulators
#pragma unroll
            for (int r = 0; r < kTabRows; ++r) {
                float t0 = ac[r][0] + ac[r][1]; ac[r][1] = ac[r][1] - (t0 - ac[r][0]); ac[r][0] = t0;
                float t1 = ac[r][2] + ac[r][3]; ac[r][3] = ac[r][3] - (t1 - ac[r][2]); ac[r][2] = t1;
            }
        }
    }
#pragma unroll
    for (int r = 0; r < kTabRows; ++r) {
        const int g = g0 + 2 * r;
        if (g > G) break;
        const float tr = ac[r][0] + ac[r][1], ti = ac[r][2] + ac[r][3];
        const dfl re = {tr, ac[r][1] - (tr - ac[r][0])}, im = {ti, ac[r][3] - (ti - ac[r][2])};
        tab[(long long)(g + G) * J + p] = make_float4(re.hi, im.hi, re.lo, im.lo);
        // D_p(-y) = conj(D_p(y)) + (-1)^p (sinc(y - h) - sinc(y + h)): m and -m
        // swap, c_{-m} = conj(c_m), and the end terms m = -h, h differ; at
        // y = g/2, sinc(y -+ h) = (-1)^h sin(pi y) / (pi (y -+ h))
        const double y = 0.5 * (double)g, sy = (g & 3) == 1 ? 1.0 : -1.0;
        const double corr = ((h & 1) ? -sy : sy) * 2.0 * (double)h / (kPi * (y * y - (double)h * (double)h));
        const dfl c = df_split((p & 1) ? -corr : corr);
        const dfl rn = df_addq(re, c);
        tab[(long long)(G - g) * J + p] = make_float4(rn.hi, -im.hi, rn.lo, -im.lo);
    }
}

// Bytes of the per-window arrays of weights_kernel (y, sin(pi y) or the far
// prefactor, three double-float and three int arrays), rounded to 16.
__host__ __device__ inline size_t weights_smem_head(int K) {
    return ((size_t)K * (2 * sizeof(double) + 3 * sizeof(float2) + 3 * sizeof(int)) + 15) & ~(size_t)15;
}

constexpr float kInv2PiHi = (float)(0.5 / kPi);
constexpr float kInv2PiLo = (float)(0.5 / kPi - (double)kInv2PiHi);

// Far windows (|y| >= 1.25 h): the ratio rho and prefactor of the Chebyshev
// expansion, its truncation R and the number R1 of leading terms taken in
// double-float (from binary32 logarithms: term counts, not values).
__device__ __forceinline__ void far_window(double y, int h, double scale, double &rho, double &f, int &R, int &R1) {
    const double a = y / (double)h;
    const double sq = copysign(sqrt((a - 1.0) * (a + 1.0)), a);
    rho = 1.0 / (a + sq);
    const float lr = -logf(fabsf((float)rho));
    R = max(1, min((int)ceilf(48.f * 0.693147181f / lr), kFarTerms));
    R1 = max(1, min((int)ceilf((25.f * 0.693147181f + logf((float)R)) / lr), R));
    f = scale * sinpi(y) * 2.0 / (kPi * (double)h * sq);
}

// G = (mu_p / 2 pi) q, mu_p / 2 pi = 1/(2 pi) or 1/pi, in double-float; the planes
// hold (Re G, -Im G).
__device__ __forceinline__ void store_weight(int J, int p, int t, int n_T, int pitch_T, dfl q, dfl qi, double *Gr,
                                             double *Gm, float2 *Gs) {
    const bool edge = p == 0 || p == J - 1;
    const dfl c = edge ? dfl{kInv2PiHi, kInv2PiLo} : dfl{2.f * kInv2PiHi, 2.f * kInv2PiLo};
    const dfl a = df_mulq(q, c), b = df_negq(df_mulq(qi, c));
    if (Gs) {
        Gs[(long long)p * pitch_T + t] = make_float2(a.hi, a.lo);
        Gs[(long long)(J + p) * pitch_T + t] = make_float2(b.hi, b.lo);
    } else {
        Gr[(long long)p * n_T + t] = (double)a.hi + (double)a.lo;
        Gm[(long long)p * n_T + t] = (double)b.hi + (double)b.lo;
    }
}

// Weights from the sampled near sums (J <= kSincTabMaxJ).  One CTA per time and
// 256 columns p, in two groups of 128 threads with two columns each; group g
// takes the windows k = g mod 2, and the groups' sums are added in order (a
// fixed split, so that a time's weights do not depend on the other times).
// Near windows: 42 samples around y, their weights (with 2W/M) formed by the
// group's first threads; far windows: Horner's rule over the far table, the
// terms past R1 in binary32.  (re, im) are one packed pair throughout.
// With many times the FMA pipe is active 60 % of the cycles and most other stalls
// wait for the table's rows out of L2; with few, the dependent steps of a window
// (weights, barrier, loads) bound it, which the groups take side by side.
// (Four groups, 512 threads, were 4 % slower with many times: fewer CTAs hide
// the FP64 set-up.)  Measured (GB300): 4096 times, J = 256, 29 windows: 0.63 ms before; 16
// times, J = 128, 7 windows: 56 us before (one window after another, re and im
// apart).
constexpr int kWGroups = 2, kWCols = 128, kWChunk = 64;

struct FarNear {
    int R, R1;          // R = 0: near
    SincPoint pt;       // near
    dfv rho, f;         // far
};

__global__ void __launch_bounds__(kWGroups *kWCols, 4) weights_tab_kernel(
    int J, int M, double W, int K, const double *__restrict__ s, const float4 *__restrict__ Bf,
    const float4 *__restrict__ nu_f, const float4 *__restrict__ tab, int G, const double *__restrict__ T, int n_T,
    double *__restrict__ Gr, double *__restrict__ Gm, float2 *__restrict__ Gs, int pitch_T) {
    __shared__ FarNear win[kWChunk];
    __shared__ float2 swt[kWGroups][kSincPts];
    __shared__ float4 part[kWGroups - 1][2 * kWCols];
    const int t = blockIdx.x, h = M / 2;
    const int grp = threadIdx.x / kWCols, lane = threadIdx.x % kWCols;
    const int p0 = blockIdx.y * 2 * kWCols + lane;
    const bool two = blockIdx.y * 2 * kWCols + kWCols < J;      // the CTA has second columns
    const int pa = min(p0, J - 1), pb = min(p0 + kWCols, J - 1);   // (columns past J - 1 are computed and dropped)
    const double tt = T[t], scale = 2.0 * W / (double)M;
    const dfv sc = df_from(scale);
    float2 qh[2], ql[2];
    qh[0] = qh[1] = ql[0] = ql[1] = p2(0.f, 0.f);
    for (int k0 = 0; k0 < K; k0 += kWChunk) {
        __syncthreads();
        for (int k = threadIdx.x; k < min(kWChunk, K - k0); k += blockDim.x) {
            FarNear w;
            const double y = W * (tt - s[k0 + k]) * (1.0 / kPi);
            w.R = w.R1 = 0;
            w.rho = w.f = df_make(0.f, 0.f);
            w.pt = SincPoint{0, 0, w.rho, w.rho};
            if (fabs(y) < 1.25 * (double)h) {
                w.pt = sinc_point(y);
            } else {
                double rho, f;
                far_window(y, h, scale, rho, f, w.R, w.R1);
                w.rho = df_from(rho);
                w.f = df_from(f);
            }
            win[k] = w;
        }
        __syncthreads();
        for (int k = k0 + grp; k < min(k0 + kWChunk, K); k += kWGroups) {
            const FarNear &w = win[k - k0];
            df2 d[2];
            if (w.R == 0) {
                asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(kWCols) : "memory");   // the last window's weights are read
                if (lane < kSincPts) {
                    const dfv v = df_mul(sinc_weight(w.pt, lane), sc);
                    swt[grp][lane] = p2(v.hi, v.lo);
                }
                asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(kWCols) : "memory");
                const float4 *row = tab + (long long)(w.pt.g0 + G) * J;
                float2 ah = p2(0.f, 0.f), al = ah, bh = ah, bl = ah;
#pragma unroll 6
                for (int q = 0; q < kSincPts; ++q) {
                    const float2 wt = swt[grp][q];
                    const df2 ww = {p2(wt.x, wt.x), p2(wt.y, wt.y)};
                    const float4 va = __ldg(row + (long long)q * J + pa);
                    df2_acc(ah, al, ww, {p2(va.x, va.y), p2(va.z, va.w)});
                    if (two) {
                        const float4 vb = __ldg(row + (long long)q * J + pb);
                        df2_acc(bh, bl, ww, {p2(vb.x, vb.y), p2(vb.z, vb.w)});
                    }
                }
                d[0] = df2_quick(ah, al);
                d[1] = df2_quick(bh, bl);
            } else {
                const float2 rh = p2(w.rho.hi, w.rho.hi), rl = p2(w.rho.lo, w.rho.lo);
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    if (c == 1 && !two) break;
                    const float4 *col = nu_f + (c ? pb : pa);
                    float2 a = p2(0.f, 0.f);
#pragma unroll 4
                    for (int r = w.R - 1; r >= w.R1; --r) {     // binary32 tail
                        const float4 v = __ldg(col + (long long)r * J);
                        a = p2_fma(a, rh, p2(v.x, v.y));
                    }
                    df2 f = {a, p2(0.f, 0.f)};
#pragma unroll 4
                    for (int r = w.R1 - 1; r >= 0; --r) {
                        const float4 v = __ldg(col + (long long)r * J);
                        float2 e;
                        const float2 x = p2_prod(f, {rh, rl}, e), vh = p2(v.x, v.y), y = p2_add(x, vh);
                        f = df2_quick(y, p2_add(p2_two_sum_err(x, vh, y), p2_add(e, p2(v.z, v.w))));
                    }
                    d[c] = df2_mul(f, df2_bcast(w.f));
                }
            }
#pragma unroll
            for (int c = 0; c < 2; ++c) {   // q += b d (complex)
                if (c == 1 && !two) break;
                const float4 b4 = __ldg(Bf + (long long)k * J + (c ? pb : pa));
                df2_acc(qh[c], ql[c], {p2(b4.x, b4.x), p2(b4.y, b4.y)}, d[c]);
                df2_acc(qh[c], ql[c], {p2(-b4.z, b4.z), p2(-b4.w, b4.w)}, df2_swap(d[c]));
            }
        }
    }
    if (grp > 0) {
#pragma unroll
        for (int c = 0; c < 2; ++c) part[grp - 1][lane + c * kWCols] = make_float4(qh[c].x, qh[c].y, ql[c].x, ql[c].y);
    }
    __syncthreads();
    if (grp > 0) return;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const int p = p0 + c * kWCols;
        if (p >= J) break;
        df2 q = df2_quick(qh[c], ql[c]);
        for (int g = 0; g < kWGroups - 1; ++g) {
            const float4 v = part[g][lane + c * kWCols];
            q = df2_add(q, {p2(v.x, v.y), p2(v.z, v.w)});
        }
        store_weight(J, p, t, n_T, pitch_T, {q.h.x, q.l.x}, {q.h.y, q.l.y}, Gr, Gm, Gs);
    }
}

// Weights without the sampled table (larger J, or no memory for it): one CTA
// per time, thread p.  The per-window quantities that do not depend on p (y,
// near or far, sin(pi y), the far ratio and its truncation R) are formed once
// per CTA.  Near windows: the direct M-term sums (near_sum); far windows:
// Horner's rule in double-float over the far table.
__global__ void __launch_bounds__(256) weights_kernel(
    int J, int M, double W, int K, const double *__restrict__ s, const double2 *__restrict__ B,
    const float4 *__restrict__ Bf, const float4 *__restrict__ nu_f, const float4 *__restrict__ ph_g,
    const double *__restrict__ T, int n_T, double *__restrict__ Gr, double *__restrict__ Gm,
    float2 *__restrict__ Gs, int pitch_T) {
    extern __shared__ __align__(16) double smd[];
    double *wy = smd;                                        // K: y
    double *wf = wy + K;                                     // K: sin(pi y) (near)
    float2 *wrho = reinterpret_cast<float2 *>(wf + K);       // K: rho (far) or 2W/M (near), double-float
    float2 *wfd = wrho + K;                                  // K: far prefactor, double-float
    int *wR = reinterpret_cast<int *>(wfd + 2 * K);          // K: far terms R | R1 << 16, 0 = near
    float4 *ph4 = reinterpret_cast<float4 *>(reinterpret_cast<char *>(smd) + weights_smem_head(K));
    float4 *sc4 = ph4 + M;   // h: [0] = (S(y), S(y+h)), [j] = (S(y-j) + S(y+j), S(y-j) - S(y+j))
    const int t = blockIdx.x;
    const int p = blockIdx.y * blockDim.x + threadIdx.x;
    const int h = M / 2;
    const double tt = T[t];
    const double scale = 2.0 * W / (double)M;
    for (int q = threadIdx.x; q < M; q += blockDim.x) ph4[q] = ph_g[q];   // phases for the direct near sums
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        const double y = W * (tt - s[k]) * (1.0 / kPi);
        wy[k] = y;
        if (fabs(y) < 1.25 * (double)h) {
            wR[k] = 0;
            const dfl sd = df_split(scale);
            wrho[k] = make_float2(sd.hi, sd.lo);
            wf[k] = sinpi(y);
        } else {
            double rho, f;
            int R, R1;
            far_window(y, h, scale, rho, f, R, R1);
            wR[k] = R | (R1 << 16);
            const dfl rr = df_split(rho), fd = df_split(f);
            wrho[k] = make_float2(rr.hi, rr.lo);
            wfd[k] = make_float2(fd.hi, fd.lo);
        }
    }
    __syncthreads();
    // G accumulates in double-float: q += B_k(w_p) D_p(t - s_k)
    float qrh = 0.f, qrl = 0.f, qih = 0.f, qil = 0.f;
    for (int k = 0; k < K; ++k) {
        const int R = wR[k] & 0xffff, R1 = wR[k] >> 16;
        dfl dr = {0.f, 0.f}, di = {0.f, 0.f};
        if (R == 0) {          // near window (the same branch in the whole CTA)
            float rh, rl, ih, il;
            near_sum(wy[k], df_split(wf[k] * (1.0 / kPi)), h, M, p, J, ph4, sc4, rh, rl, ih, il);
            if (p < J) {
                const float2 sd = wrho[k];   // 2W/M
                dr = df_mulq({rh, rl}, {sd.x, sd.y});
                di = df_mulq({ih, il}, {sd.x, sd.y});
            }
        } else if (p < J) {
            const float2 r2 = wrho[k];
            const dfl rho = {r2.x, r2.y};
            float ah = 0.f, bh = 0.f;
            for (int r = R - 1; r >= R1; --r) {     // FP32 tail
                const float4 v = nu_f[(long long)r * J + p];
                ah = fmaf(ah, rho.hi, v.x);
                bh = fmaf(bh, rho.hi, v.y);
            }
            float al = 0.f, bl = 0.f;
            for (int r = R1 - 1; r >= 0; --r) {
                const float4 v = nu_f[(long long)r * J + p];
                df_horner(ah, al, rho, v.x, v.z);
                df_horner(bh, bl, rho, v.y, v.w);
            }
            const float2 f2 = wfd[k];
            const dfl f = {f2.x, f2.y};
            dr = df_mulq({ah, al}, f);
            di = df_mulq({bh, bl}, f);
        }
        if (p < J) {
            dfl br, bi;
            if (Bf) {
                const float4 b4 = Bf[(long long)k * J + p];
                br = {b4.x, b4.y};
                bi = {b4.z, b4.w};
            } else {
                const double2 b = B[(long long)k * J + p];
                br = df_split(b.x);
                bi = df_split(b.y);
            }
            // q += b * d (complex)
            df_mac(qrh, qrl, br, dr);
            df_mac(qrh, qrl, {-bi.hi, -bi.lo}, di);
            df_mac(qih, qil, br, di);
            df_mac(qih, qil, bi, dr);
        }
    }
    if (p < J) store_weight(J, p, t, n_T, pitch_T, {qrh, qrl}, {qih, qil}, Gr, Gm, Gs);
}

constexpr int BM = 64, BN = 64, BK = 16;

// u[x][t] = sum_{kk < 2J} A[x][kk] Bm[kk][t], A = [Vr | Vi], Bm = [Gr ; Gm].
// For sums that contract_slices_fp64 does not take (up to 2^25 products, 2J >
// 8192, scratch) and the synthesis without allocation.
// kTile x kTile outputs per CTA, (kTile / 16)^2 per thread.  Bound by the FP64
// pipe (1.19 of the 1.25 TFLOP/s that FMA chains reach at 1024 x 4096, 2J = 512), so
// what matters is that every SM has a tile: tiles of 32 where tiles of 64 are
// fewer than two per SM (333 x 1001, 2J = 402: 96 tiles, 0.50 ms).
template <int kTile>
__global__ void __launch_bounds__(256) contract_kernel(int J, int n_x, int n_T,
                                                       const double2 *__restrict__ V,
                                                       const double *__restrict__ Gr,
                                                       const double *__restrict__ Gm,
                                                       double *__restrict__ u) {
    constexpr int kPer = kTile / 16;
    __shared__ double As[BK][kTile];
    __shared__ double Bs[BK][kTile + 2];
    const int x0 = blockIdx.y * kTile, t0 = blockIdx.x * kTile;
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    double acc[kPer][kPer] = {};
    const int K2 = 2 * J;
    for (int k0 = 0; k0 < K2; k0 += BK) {
        for (int e = tid; e < BK * kTile; e += 256) {
            const int kk = e / kTile, xx = e % kTile;
            const int k = k0 + kk, x = x0 + xx;
            double v = 0.0;
            if (k < K2 && x < n_x) {
                const double2 vv = V[(long long)(k < J ? k : k - J) * n_x + x];
                v = (k < J) ? vv.x : vv.y;
            }
            As[kk][xx] = v;
        }
        for (int e = tid; e < BK * kTile; e += 256) {
            const int kk = e / kTile, tt = e % kTile;
            const int k = k0 + kk, t = t0 + tt;
            double v = 0.0;
            if (k < K2 && t < n_T) v = (k < J) ? Gr[(long long)k * n_T + t] : Gm[(long long)(k - J) * n_T + t];
            Bs[kk][tt] = v;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            double a[kPer], b[kPer];
#pragma unroll
            for (int i = 0; i < kPer; ++i) a[i] = As[kk][ty * kPer + i];
#pragma unroll
            for (int j = 0; j < kPer; ++j) b[j] = Bs[kk][tx * kPer + j];
#pragma unroll
            for (int i = 0; i < kPer; ++i)
#pragma unroll
                for (int j = 0; j < kPer; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int x = x0 + ty * kPer + i;
        if (x >= n_x) continue;
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int t = t0 + tx * kPer + j;
            if (t < n_T) u[(long long)x * n_T + t] = acc[i][j];
        }
    }
}

// The same sums for few outputs (contract_small): CTAs of 8 targets x 16 times,
// a warp per four times and slice of the frequencies, lane = (target, every
// fourth frequency of the slice), so that a few thousand outputs spread over
// the chip and nothing is staged; the slices are summed in order.  With fewer
// than two CTAs per SM the latency of a lane's loads bounds it: four slices, a
// quarter of the loads in a row.  Measured (GB300), one slice -> four: 777
// targets x 16 times, 2J = 256 18.5 -> 12.4 us (66 us through the tensor-core
// contraction's launches), 30 x 64, 2J = 1024 59.6 -> 37.0 us; 4000 x 16, 2J =
// 128 (500 CTAs, FP64 pipe) 20.6 -> 24.7 us.
template <int kSmallSlices>
__global__ void __launch_bounds__(128 * kSmallSlices) contract_small_kernel(
    int J, int n_x, int n_T, const double2 *__restrict__ V, const double *__restrict__ Gr,
    const double *__restrict__ Gm, double *__restrict__ u) {
    __shared__ double part[kSmallSlices][16][8 + 1];
    const int x_tiles = (n_x + 7) / 8, x0 = (int)(blockIdx.x % x_tiles) * 8, t0 = (int)(blockIdx.x / x_tiles) * 16;
    const int lane = threadIdx.x & 31, x = x0 + (lane & 7);
    const int tg = (threadIdx.x >> 5) & 3, slice = threadIdx.x >> 7;
    int tt[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) tt[i] = min(t0 + 4 * tg + i, n_T - 1);
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    if (t0 + 4 * tg < n_T) {   // whole warps
#pragma unroll 4
        for (int p = 4 * slice + (lane >> 3); p < J; p += 4 * kSmallSlices) {
            const double2 v = x < n_x ? __ldg(V + (long long)p * n_x + x) : make_double2(0.0, 0.0);
            const double *gr = Gr + (long long)p * n_T, *gm = Gm + (long long)p * n_T;
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i] = fma(v.x, __ldg(gr + tt[i]), fma(v.y, __ldg(gm + tt[i]), acc[i]));
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], 8);
            acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], 16);
            if (lane < 8) part[slice][4 * tg + i][lane] = acc[i];
        }
    }
    __syncthreads();
    const int q = threadIdx.x & 15, r = threadIdx.x >> 4;   // time, target (the first 128 threads)
    if (r < 8 && x0 + r < n_x && t0 + q < n_T) {
        double v = part[0][q][r];
#pragma unroll
        for (int i = 1; i < kSmallSlices; ++i) v += part[i][q][r];
        u[(long long)(x0 + r) * n_T + t0 + q] = v;
    }
}

// V[j][x] (complex FP64) as double-float rows of the contraction's left
// operand: row j holds the real parts, row J + j the imaginary parts (row
// pitch px, a multiple of 4).
__global__ void split_v_kernel(int J, int n_x, int px, const double2 *__restrict__ V,
                               float2 *__restrict__ Vs) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (x >= px) return;
    float2 r = make_float2(0.f, 0.f), i = r;
    if (x < n_x) {
        const double2 v = V[(long long)j * n_x + x];
        const dfl a = df_split(v.x), b = df_split(v.y);
        r = make_float2(a.hi, a.lo);
        i = make_float2(b.hi, b.lo);
    }
    Vs[(long long)j * px + x] = r;
    Vs[(long long)(J + j) * px + x] = i;
}

// The contraction in double-float arithmetic (mixed-precision paths):
//   u[x][t] = sum_{kk < 2J} Vs[kk][x] Gs[kk][t],
// both operands double-float pairs (hi, lo) with rows along x and t.  Each
// product is formed exactly (FMA residual) plus the hi*lo cross terms and
// every output accumulates as a double-float pair (two-sum), ~2^-44 relative
// per step.  64 x 64 outputs per CTA, 4 x 4 per thread (t in two pairs 32
// apart, so that shared-memory reads of a warp are contiguous); the next
// 16-deep slice of both operands is loaded into registers while the current
// one is consumed from shared memory (two buffers, one barrier per slice).
// Operand elements past n_x, n_T or 2J are read as zero.
__global__ void __launch_bounds__(256) contract_df_kernel(int J, int n_x, int n_T, int px, int pt,
                                                          const float2 *__restrict__ Vs,
                                                          const float2 *__restrict__ Gs,
                                                          double *__restrict__ u) {
    __shared__ __align__(16) float2 As[2][BK][BM];
    __shared__ __align__(16) float2 Bs[2][BK][BN];
    const int x0 = blockIdx.y * BM, t0 = blockIdx.x * BN;
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    const int K2 = 2 * J;
    float sh[4][4], sl[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) sh[i][j] = sl[i][j] = 0.f;

    // slice loader: element e = tid + 256 h (h = 0, 1) is row e / 32, float2
    // pair e % 32 of the 16 x 64 slice
    float4 ra[2], rb[2];
    auto load = [&](int k0) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = tid + 256 * h, kk = k0 + (e >> 5), c = 2 * (e & 31);
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
            if (kk < K2) {
                const int x = x0 + c, t = t0 + c;
                if (x < n_x) {
                    a = __ldg(reinterpret_cast<const float4 *>(Vs + (long long)kk * px + x));
                    if (x + 1 >= n_x) a.z = a.w = 0.f;
                }
                if (t < n_T) {
                    b = __ldg(reinterpret_cast<const float4 *>(Gs + (long long)kk * pt + t));
                    if (t + 1 >= n_T) b.z = b.w = 0.f;
                }
            }
            ra[h] = a;
            rb[h] = b;
        }
    };
    auto store = [&](int buf) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = tid + 256 * h, kk = e >> 5, c = 2 * (e & 31);
            *reinterpret_cast<float4 *>(&As[buf][kk][c]) = ra[h];
            *reinterpret_cast<float4 *>(&Bs[buf][kk][c]) = rb[h];
        }
    };
    load(0);
    store(0);
    __syncthreads();
    int buf = 0;
    for (int k0 = 0; k0 < K2; k0 += BK) {
        const bool more = k0 + BK < K2;
        if (more) load(k0 + BK);
#pragma unroll 4
        for (int kk = 0; kk < BK; ++kk) {
            float2 a[4], b[4];
            const float4 a01 = *reinterpret_cast<const float4 *>(&As[buf][kk][ty * 4]);
            const float4 a23 = *reinterpret_cast<const float4 *>(&As[buf][kk][ty * 4 + 2]);
            const float4 b01 = *reinterpret_cast<const float4 *>(&Bs[buf][kk][tx * 2]);
            const float4 b23 = *reinterpret_cast<const float4 *>(&Bs[buf][kk][32 + tx * 2]);
            a[0] = make_float2(a01.x, a01.y);
            a[1] = make_float2(a01.z, a01.w);
            a[2] = make_float2(a23.x, a23.y);
            a[3] = make_float2(a23.z, a23.w);
            b[0] = make_float2(b01.x, b01.y);
            b[1] = make_float2(b01.z, b01.w);
            b[2] = make_float2(b23.x, b23.y);
            b[3] = make_float2(b23.z, b23.w);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float pp = a[i].x * b[j].x;
                    float pe = fmaf(a[i].x, b[j].x, -pp);
                    pe = fmaf(a[i].x, b[j].y, pe);
                    pe = fmaf(a[i].y, b[j].x, pe);
                    const float t = sh[i][j] + pp;
                    const float z = t - sh[i][j];
                    sl[i][j] += ((sh[i][j] - (t - z)) + (pp - z)) + pe;
                    sh[i][j] = t;
                }
        }
        if (more) store(buf ^ 1);
        __syncthreads();
        buf ^= 1;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int x = x0 + ty * 4 + i;
        if (x >= n_x) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int t = t0 + (j < 2 ? tx * 2 + j : 32 + tx * 2 + (j - 2));
            if (t < n_T) u[(long long)x * n_T + t] = (double)sh[i][j] + (double)sl[i][j];
        }
    }
}

}  // namespace

void launch_far_table(int J, int M, double *pw, double2 *nu, float4 *nu_f, float4 *phase_tab,
                      cudaStream_t st) {
    far_powers_kernel<<<(M + 127) / 128, 128, 0, st>>>(M, pw);
    far_table_kernel<<<J, 128, 0, st>>>(J, M, pw, nu, nu_f, phase_tab);
}

void launch_sinc_table(int J, int M, const float4 *phase_tab, float4 *tab, cudaStream_t st) {
    const int G = sinc_tab_half(J);
    if (!G) return;
    const size_t smem = (size_t)(M + kTabRows * (M / 2)) * sizeof(float4);
    static std::atomic<unsigned long long> attr{0};
    ensure_smem_attr((const void *)sinc_table_kernel, 200 * 1024, attr);
    const int odd_ctas = ((G + 1) / 2 + kTabRows - 1) / kTabRows;   // positive odd rows 1 .. G
    sinc_table_kernel<<<dim3(odd_ctas + 64, (J + kTabThreads - 1) / kTabThreads), kTabThreads, smem, st>>>(
        J, M, G, odd_ctas, phase_tab, tab);
}

size_t synth_weights_smem(int J, int K, bool table) {
    const int M = 2 * (J - 1);
    return weights_smem_head(K) + (table ? 0 : (size_t)(M + M / 2) * sizeof(float4));
}

void launch_synth_weights(int J, int M, double W, int K, const double *s, const double2 *B,
                          const float4 *Bf, const float4 *nu_f, const float4 *phase_tab,
                          const float4 *sinc_tab, const double *T, int n_T, double *Gr, double *Gm,
                          float2 *Gs, cudaStream_t st) {
    if (n_T <= 0) return;
    if (sinc_tab) {
        weights_tab_kernel<<<dim3(n_T, (J + 2 * kWCols - 1) / (2 * kWCols)), kWGroups * kWCols, 0, st>>>(
            J, M, W, K, s, Bf, nu_f, sinc_tab, sinc_tab_half(J), T, n_T, Gr, Gm, Gs, synth_pitch(n_T));
        return;
    }
    const size_t smem = synth_weights_smem(J, K, false);
    static std::atomic<unsigned long long> attr{0};
    ensure_smem_attr((const void *)weights_kernel, (int)kWeightsMaxSmem, attr);
    weights_kernel<<<dim3(n_T, (J + 255) / 256), 256, smem, st>>>(J, M, W, K, s, B, Bf, nu_f, phase_tab, T, n_T, Gr, Gm,
                                                                 Gs, synth_pitch(n_T));
}

void launch_synth_contract(int J, int n_x, int n_T, const double2 *V, const double *Gr,
                           const double *Gm, double *u, cudaStream_t st) {
    if (n_x <= 0 || n_T <= 0) return;
    auto tiles = [&](int e) { return dim3((n_T + e - 1) / e, (n_x + e - 1) / e); };
    const dim3 g64 = tiles(64);
    if (contract_small(J, n_x, n_T)) {
        // all tiles in grid.x: J = 2 leaves 2^22 outputs, which for one target are more than 65535 tiles of 16 times
        const unsigned ctas = (unsigned)((n_x + 7) / 8) * (unsigned)((n_T + 15) / 16);
        if (ctas < 2 * kSms)
            contract_small_kernel<4><<<ctas, 4 * 128, 0, st>>>(J, n_x, n_T, V, Gr, Gm, u);
        else
            contract_small_kernel<1><<<ctas, 128, 0, st>>>(J, n_x, n_T, V, Gr, Gm, u);
    } else if (g64.x * g64.y < 2 * kSms)
        contract_kernel<32><<<tiles(32), 256, 0, st>>>(J, n_x, n_T, V, Gr, Gm, u);
    else
        contract_kernel<64><<<g64, 256, 0, st>>>(J, n_x, n_T, V, Gr, Gm, u);
}

void launch_synth_contract_df(int J, int n_x, int n_T, const double2 *V, float2 *Vs,
                              const float2 *Gs, double *u, cudaStream_t st) {
    if (n_x <= 0 || n_T <= 0) return;
    const int px = synth_pitch(n_x), pt = synth_pitch(n_T);
    split_v_kernel<<<dim3((px + 255) / 256, J), 256, 0, st>>>(J, n_x, px, V, Vs);
    dim3 grid((n_T + BN - 1) / BN, (n_x + BM - 1) / BM);
    contract_df_kernel<<<grid, 256, 0, st>>>(J, n_x, n_T, px, pt, Vs, Gs, u);
}

}  // namespace fh
