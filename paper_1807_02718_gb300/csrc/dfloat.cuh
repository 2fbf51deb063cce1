// Double-float ("df") arithmetic on the FP32 pipe, and the Hankel-form
// Bessel functions of orders 0 and 1 at x >= 8 evaluated with it.
//
// A df value is hi + lo with |lo| <= ulp(hi) / 2, ~2^-48 relative.  Products
// use the exact FMA residual (two-product), sums Knuth's two-sum; each
// operation is accurate to a few 2^-46 relative.  FP32 issues 64 times as
// many operations per clock as FP64 on this GPU, so a df operation (5-15
// FP32 instructions) costs a fraction of one FP64 instruction's issue slot.
//
// Hankel form (x >= 8, A&S 9.2.5-9.2.6, 9.2.9-9.2.10):
//   H_nu(x) = sqrt(2/(pi x)) (P_nu + i Q_nu) e^{i (x - (2 nu + 1) pi/4)},
//   P0 = 1 - 9u/8192 + u^2 G0,   Q0 = (8/x)(-1/64 + 75u/524288 + u^2 G1),
//   P1 = 1 + 15u/8192 + u^2 G2,  Q1 = (8/x)(3/64 - 105u/524288 + u^2 G3),
// u = (8/x)^2.  The leading coefficients are exact binary32 numbers; each
// remainder u^2 G_k (|.| <= 1e-4) is a polynomial whose constant term is a
// df pair and whose other terms (|.| <= 1e-6) are binary32 (bessel_cheb.h),
// so the df results carry ~1e-14 absolute error.
#pragma once

#include "bessel_cheb.h"

namespace fh {

struct dfv {
    float hi, lo;
};

__device__ __forceinline__ dfv df_make(float hi, float lo) { return {hi, lo}; }

__device__ __forceinline__ dfv df_from(double v) {
    const float h = (float)v;
    return {h, (float)(v - (double)h)};
}

__device__ __forceinline__ double df_to(dfv a) { return (double)a.hi + (double)a.lo; }

// A complex FP64 value as double-float pairs (re hi, re lo, im hi, im lo).
__device__ __forceinline__ float4 df_pack(double re, double im) {
    const dfv r = df_from(re), i = df_from(im);
    return make_float4(r.hi, r.lo, i.hi, i.lo);
}

__device__ __forceinline__ dfv df_quick(float s, float e) {   // |s| >= |e|
    const float h = s + e;
    return {h, e - (h - s)};
}

__device__ __forceinline__ dfv df_add(dfv a, dfv b) {
    const float s = a.hi + b.hi;
    const float bb = s - a.hi;
    const float e = ((a.hi - (s - bb)) + (b.hi - bb)) + (a.lo + b.lo);
    return df_quick(s, e);
}

__device__ __forceinline__ dfv df_add_f(dfv a, float b) {
    const float s = a.hi + b;
    const float bb = s - a.hi;
    const float e = ((a.hi - (s - bb)) + (b - bb)) + a.lo;
    return df_quick(s, e);
}

__device__ __forceinline__ dfv df_neg(dfv a) { return {-a.hi, -a.lo}; }

__device__ __forceinline__ dfv df_mul(dfv a, dfv b) {
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return df_quick(p, e);
}

__device__ __forceinline__ dfv df_mul_f(dfv a, float b) {
    const float p = a.hi * b;
    const float e = fmaf(a.lo, b, fmaf(a.hi, b, -p));
    return df_quick(p, e);
}

// a * b + c

// a * b + c with one renormalisation: the exact product of the hi parts (FMA
// residual) and the cross terms, the sum of the two leading parts by two-sum,
// every small part added into one error term.
__device__ __forceinline__ dfv df_mad(dfv a, dfv b, dfv c) {
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    const float s = p + c.hi;
    const float bb = s - p;
    return df_quick(s, ((p - (s - bb)) + (c.hi - bb)) + (e + c.lo));
}

// a * b + c * d with one renormalisation (two exact products, one two-sum).
__device__ __forceinline__ dfv df_dot2(dfv a, dfv b, dfv c, dfv d) {
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    const float q = c.hi * d.hi;
    float f = fmaf(c.hi, d.hi, -q);
    f = fmaf(c.hi, d.lo, f);
    f = fmaf(c.lo, d.hi, f);
    const float s = p + q;
    const float bb = s - p;
    return df_quick(s, ((p - (s - bb)) + (q - bb)) + (e + f));
}

__device__ __forceinline__ dfv df_sqrt(dfv a) {
    const float s = sqrtf(a.hi);
    const float e = (fmaf(-s, s, a.hi) + a.lo) * (0.5f / s);
    return df_quick(s, e);
}

__device__ __forceinline__ dfv df_rcp(dfv a) {
    const float r = 1.0f / a.hi;
    const float t = fmaf(-a.hi, r, 1.0f) - a.lo * r;   // 1 - a r
    return df_quick(r, r * t);
}

// sin and cos of a df argument |y| <= pi/4 (Taylor series to degree 17 / 16,
// truncation < 2^-53).  Horner in y^2; the coefficients of y^12 and beyond
// (<= 1/12! = 2.1e-9, times y^12 <= 0.055) need only binary32, the rest are
// df multiply-adds.
__device__ __forceinline__ void df_sincos_small(dfv y, dfv &sn, dfv &cs) {
    const dfv y2 = df_mul(y, y);
    float ts = kSinDF[16], tc = kCosDF[16];
#pragma unroll
    for (int k = 7; k >= 6; --k) {
        ts = fmaf(ts, y2.hi, kSinDF[2 * k]);
        tc = fmaf(tc, y2.hi, kCosDF[2 * k]);
    }
    dfv ps = df_make(ts, 0.f), pc = df_make(tc, 0.f);
#pragma unroll
    for (int k = 5; k >= 0; --k) {
        ps = df_mad(ps, y2, df_make(kSinDF[2 * k], kSinDF[2 * k + 1]));
        pc = df_mad(pc, y2, df_make(kCosDF[2 * k], kCosDF[2 * k + 1]));
    }
    sn = df_mul(ps, y);
    cs = pc;
}

// e^{i y} for a double-float 0 <= y < 3.1 without FP64: the Taylor series at
// y / 2^h with y / 2^h <= 0.78 (h = 0, 1 or 2; halving is exact), then h
// double-angle steps cos 2a = 1 - 2 sin^2 a, sin 2a = 2 sin a cos a.  The
// frequency step e^{i dkappa r} of the wide-band fields reaches y ~ 1.6.
__device__ __forceinline__ void df_sincos_mid(dfv y, dfv &sn, dfv &cs) {
    const int h = (y.hi >= 0.78f) + (y.hi >= 1.56f);
    const float sc = h == 0 ? 1.f : h == 1 ? 0.5f : 0.25f;
    df_sincos_small(df_make(y.hi * sc, y.lo * sc), sn, cs);
    for (int k = 0; k < h; ++k) {
        const dfv s2 = df_mul(sn, sn);
        const dfv c2 = df_add_f(df_mul_f(s2, -2.f), 1.f);
        sn = df_mul_f(df_mul(sn, cs), 2.f);
        cs = c2;
    }
}

// e^{i x} for an FP64 argument 0 <= x < 2^20: quadrant reduction in FP64 (two
// FMAs with pi/2 split into two doubles), the rest in df.
__device__ __forceinline__ void df_expi(double x, dfv &c, dfv &s) {
    constexpr double kPio2Hi = 1.5707963267948966192;
    constexpr double kPio2Lo = 6.123233995736766036e-17;
    const double k = rint(x * 0.63661977236758134308);
    double y = fma(-k, kPio2Hi, x);
    y = fma(-k, kPio2Lo, y);
    dfv sn, cs;
    df_sincos_small(df_from(y), sn, cs);
    const int q = ((int)k) & 3;
    if (q == 0) { c = cs; s = sn; }
    else if (q == 1) { c = df_neg(sn); s = cs; }
    else if (q == 2) { c = df_neg(cs); s = df_neg(sn); }
    else { c = sn; s = df_neg(cs); }
}

// e^{i (x - pi/4)} for x = kappa r, kappa = k1 + k2 + k3 (three binary32
// pieces, exact for an FP64 kappa), r double-float, 0 <= k1 r.hi < kExpiKrMax.
// x - pi/4 - q pi/2 is formed without rounding x first (Cody-Waite with pi/2 =
// C1 + C2 + C3): k1 r.hi - q C1 exactly (FMA residual; q C1 exact and the
// difference exact by Sterbenz's lemma), the O(2^-24 x) terms k1 r.lo,
// k2 r.hi, q C2 exactly as double-float pairs, the O(2^-48 x) terms in
// binary32.  Then the Taylor series on |y| <= pi/4 and the quadrant q.
constexpr float kExpiKrMax = 6000.f;   // q < 2^12, so that q C1 is exact

__device__ __forceinline__ void df_expi_kr(float k1, float k2, float k3, dfv r, dfv &c, dfv &s) {
    const float p1 = k1 * r.hi;
    const float e1 = fmaf(k1, r.hi, -p1);
    const float qf = rintf((p1 - kPio4DF[0]) * 0.636619772f);
    const float y0 = fmaf(-qf, kPio2CW[0], p1);
    const float a = k1 * r.lo, ae = fmaf(k1, r.lo, -a);
    const float b = k2 * r.hi, be = fmaf(k2, r.hi, -b);
    const float m = qf * kPio2CW[1], me = fmaf(qf, kPio2CW[1], -m);
    dfv t = df_add(df_make(a, ae), df_make(b, be));
    t = df_add(t, df_make(-m, -me));
    t = df_add(t, df_make(-kPio4DF[0], -kPio4DF[1]));
    t = df_add_f(t, e1);
    const float tail = fmaf(k2, r.lo, fmaf(k3, r.hi, -qf * kPio2CW[2]));
    const dfv y = df_add_f(df_add(df_make(y0, 0.f), t), tail);
    dfv sn, cs;
    df_sincos_small(y, sn, cs);
    const int q = ((int)qf) & 3;
    if (q == 0) { c = cs; s = sn; }
    else if (q == 1) { c = df_neg(sn); s = cs; }
    else if (q == 2) { c = df_neg(cs); s = df_neg(sn); }
    else { c = sn; s = df_neg(cs); }
}

// ---- two double-float values at once ----
// The packed binary32 instructions (two FMAs, products or sums on a register
// pair) leave the FMA pipe's rate as it is (measured: 75 against 74 TFLOP/s)
// but take one issue slot for two operations, and issue is what bounds the
// kernels below.  Each function is the scalar one applied to both halves.
struct df2 {
    float2 h, l;
};

__device__ __forceinline__ float2 p2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 p2_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 p2_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 p2_sub(float2 a, float2 b) { return __fadd2_rn(a, p2_neg(b)); }
__device__ __forceinline__ float2 p2_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 p2_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

__device__ __forceinline__ df2 df2_make(dfv a, dfv b) { return {p2(a.hi, b.hi), p2(a.lo, b.lo)}; }
__device__ __forceinline__ dfv df2_x(df2 a) { return {a.h.x, a.l.x}; }
__device__ __forceinline__ dfv df2_y(df2 a) { return {a.h.y, a.l.y}; }
__device__ __forceinline__ df2 df2_bcast(dfv a) { return {p2(a.hi, a.hi), p2(a.lo, a.lo)}; }
__device__ __forceinline__ df2 df2_swap(df2 a) { return {p2(a.h.y, a.h.x), p2(a.l.y, a.l.x)}; }

__device__ __forceinline__ df2 df2_quick(float2 s, float2 e) {   // |s| >= |e|
    const float2 h = p2_add(s, e);
    return {h, p2_sub(e, p2_sub(h, s))};
}

__device__ __forceinline__ float2 p2_two_sum_err(float2 a, float2 b, float2 s) {   // s = a + b
    const float2 bb = p2_sub(s, a);
    return p2_add(p2_sub(a, p2_sub(s, bb)), p2_sub(b, bb));
}

__device__ __forceinline__ df2 df2_add(df2 a, df2 b) {
    const float2 s = p2_add(a.h, b.h);
    return df2_quick(s, p2_add(p2_two_sum_err(a.h, b.h, s), p2_add(a.l, b.l)));
}

__device__ __forceinline__ df2 df2_add_f(df2 a, float2 b) {
    const float2 s = p2_add(a.h, b);
    return df2_quick(s, p2_add(p2_two_sum_err(a.h, b, s), a.l));
}

// a b as the rounded product and its error with the cross terms
__device__ __forceinline__ float2 p2_prod(df2 a, df2 b, float2 &e) {
    const float2 p = p2_mul(a.h, b.h);
    e = p2_fma(a.h, b.h, p2_neg(p));
    e = p2_fma(a.h, b.l, e);
    e = p2_fma(a.l, b.h, e);
    return p;
}

__device__ __forceinline__ df2 df2_mul(df2 a, df2 b) {
    float2 e;
    const float2 p = p2_prod(a, b, e);
    return df2_quick(p, e);
}

__device__ __forceinline__ df2 df2_dot2(df2 a, df2 b, df2 c, df2 d) {   // a b + c d
    float2 e, f;
    const float2 p = p2_prod(a, b, e), q = p2_prod(c, d, f), s = p2_add(p, q);
    return df2_quick(s, p2_add(p2_two_sum_err(p, q, s), p2_add(e, f)));
}

__device__ __forceinline__ df2 df2_dot3(df2 a, df2 b, df2 c, df2 d, df2 u, df2 v) {   // a b + c d + u v
    float2 e, f, g;
    const float2 p = p2_prod(a, b, e), q = p2_prod(c, d, f), w = p2_prod(u, v, g), s = p2_add(p, q), t = p2_add(s, w);
    const float2 err = p2_add(p2_two_sum_err(p, q, s), p2_two_sum_err(s, w, t));
    return df2_quick(t, p2_add(err, p2_add(p2_add(e, f), g)));
}

// sum += a b: the product's error and the cross terms enter the low part with
// the exact two-sum error of the high part; the running sum (sh, sl) is a pair
// that the caller renormalises (df2_quick) every few terms.
__device__ __forceinline__ void df2_acc(float2 &sh, float2 &sl, df2 a, df2 b) {
    float2 e;
    const float2 p = p2_prod(a, b, e), t = p2_add(sh, p);
    sl = p2_add(sl, p2_add(p2_two_sum_err(sh, p, t), e));
    sh = t;
}

// The same with the low part compensated too: the running sum is (sh, sl, sc),
// and the product's error with the exact two-sum error of the high part enters
// sl by a second two-sum.
__device__ __forceinline__ void df2_acc_c(float2 &sh, float2 &sl, float2 &sc, df2 a, df2 b) {
    float2 e;
    const float2 p = p2_prod(a, b, e), t = p2_add(sh, p);
    const float2 x = p2_add(p2_two_sum_err(sh, p, t), e), u = p2_add(sl, x);
    sc = p2_add(sc, p2_two_sum_err(sl, x, u));
    sl = u;
    sh = t;
}

// The sum of df2_acc_c, renormalised.
__device__ __forceinline__ df2 df2_sum3(float2 sh, float2 sl, float2 sc) {
    const df2 t = df2_quick(sh, sl);
    return df2_quick(t.h, p2_add(t.l, sc));
}

// Remainder polynomials of the Hankel form for two functions at a time (which
// two: PQ0 = P0 with Q0; PP = P0 with P1 and QQ = Q0 with Q1), coefficients
// interleaved: (c1 c1' c2 c2'), (c3 c3' c4 c4'), (c5 c5' c0.hi c0'.hi), (c0.lo
// c0'.lo centre 1/half-width), so that a pair is four 16-byte loads.
template <int kPairs> struct GPair {
    float4 v[kPQ_NI][kPairs][4];
};

template <int kPairs>
__device__ __forceinline__ void g_stage_pairs(GPair<kPairs> &tb, const int (&fa)[kPairs], const int (&fb)[kPairs]) {
    for (int e = threadIdx.x; e < kPQ_NI * kPairs; e += blockDim.x) {
        const int k = e / kPairs, q = e % kPairs;
        const float *a = kG + (k * 4 + fa[q]) * kG_TERMS, *b = kG + (k * 4 + fb[q]) * kG_TERMS;
        const float *a0 = kG0DF + 2 * (k * 4 + fa[q]), *b0 = kG0DF + 2 * (k * 4 + fb[q]);
        tb.v[k][q][0] = make_float4(a[1], b[1], a[2], b[2]);
        tb.v[k][q][1] = make_float4(a[3], b[3], a[4], b[4]);
        tb.v[k][q][2] = make_float4(a[5], b[5], a0[0], b0[0]);
        tb.v[k][q][3] = make_float4(a0[1], b0[1], kPQ_UCf[k], kPQ_IUHf[k]);
    }
}

__device__ __forceinline__ int g_interval(float xf) {
    return (xf >= 10.f) + (xf >= 13.f) + (xf >= 18.f) + (xf >= 28.f) + (xf >= 60.f);
}

// u k + u^2 G with G = c0 + at (c0 a df pair, at binary32, k an exact binary32
// coefficient) for both functions: the Hankel terms of P or Q after the
// constant one.  The constant term of G and the Hankel term dominate what is
// added to them, so that a sum's error takes three operations; u2 = u^2 need
// not be renormalised.  c6 and c7 are zero on every interval
// (gen_bessel_cheb.py checks that at most six terms are needed).
__device__ __forceinline__ df2 pq_rem_pair(const float4 *g, float uhi, dfv u, float2 k, dfv u2) {
    const float4 g0 = g[0], g1 = g[1], g2 = g[2], g3 = g[3];
    const float tv = (uhi - g3.z) * g3.w;
    const float2 t = p2(tv, tv), uh = p2(u.hi, u.hi), ul = p2(u.lo, u.lo);
    float2 a = p2_fma(p2(g2.x, g2.y), t, p2(g1.z, g1.w));
    a = p2_fma(a, t, p2(g1.x, g1.y));
    a = p2_fma(a, t, p2(g0.z, g0.w));
    a = p2_mul(p2_fma(a, t, p2(g0.x, g0.y)), t);
    const float2 c0 = p2(g2.z, g2.w), gh = p2_add(c0, a);
    const float2 gl = p2_add(p2_sub(a, p2_sub(gh, c0)), p2(g3.x, g3.y));
    const float2 p = p2_mul(uh, k);
    const float2 pe = p2_fma(ul, k, p2_fma(uh, k, p2_neg(p)));
    float2 qe;
    const float2 q = p2_prod({p2(u2.hi, u2.hi), p2(u2.lo, u2.lo)}, {gh, gl}, qe);
    const float2 s = p2_add(p, q);
    return df2_quick(s, p2_add(p2_sub(q, p2_sub(s, p)), p2_add(pe, qe)));
}

// u^2 of u = (8 / x)^2 as a double-float value (not renormalised)
__device__ __forceinline__ dfv df_square(dfv u) {
    const float p = u.hi * u.hi;
    return {p, fmaf(u.hi, u.lo + u.lo, fmaf(u.hi, u.hi, -p))};
}

// Hankel form at x = kappa r >= 8, scaled by the amplitude that the caller
// carries in the phase: r8 = 8 / x, cs = a (cos, sin)(x - pi/4) for any real a,
// sc its halves exchanged; the values are a' times the Bessel functions, a' =
// a / sqrt(2 / (pi x)) (a = sqrt(2 / (pi x)) gives J and Y themselves).  P = 1 +
// dP: each value is the phase component plus one two-product dot product of
// the small corrections (|dP| <= 1.2e-3, |Q| <= 0.05).
// Order 0: (J0, Y0) = (c, s) + dP0 (c, s) + Q0 (-s, c).
__device__ __forceinline__ df2 df2_hankel0(const GPair<1> &tb, float xf, dfv r8, df2 cs, df2 sc) {
    const dfv u = df_mul(r8, r8);
    const df2 rem = pq_rem_pair(tb.v[g_interval(xf)][0], u.hi, u, p2(-9.0f / 8192.0f, 75.0f / 524288.0f), df_square(u));
    const float sq = rem.h.y - 1.0f / 64.0f;   // Q0 = r8 (rem - 1/64)
    const dfv Q0 = df_mul(r8, {sq, rem.l.y + (rem.h.y - (sq + 1.0f / 64.0f))});
    const df2 dP = {p2(rem.h.x, rem.h.x), p2(rem.l.x, rem.l.x)};
    return df2_add(cs, df2_dot2(dP, cs, {p2(-Q0.hi, Q0.hi), p2(-Q0.lo, Q0.lo)}, sc));
}

// Orders 0 and 1 together: J = (J0, J1) = (c, s) + dP (c, s) + Q m and N = -(Y0,
// Y1) = m + dP m - Q (c, s), m = (-s, c) (e^{i (x - 3 pi/4)} = (s, -c)).
__device__ __forceinline__ void df2_hankel01(const GPair<2> &tb, float xf, dfv r8, df2 cs, df2 sc, df2 &J, df2 &N) {
    const dfv u = df_mul(r8, r8), u2 = df_square(u);
    const float4 (*g)[4] = tb.v[g_interval(xf)];
    const df2 dP = pq_rem_pair(g[0], u.hi, u, p2(-9.0f / 8192.0f, 15.0f / 8192.0f), u2);
    const df2 rq = pq_rem_pair(g[1], u.hi, u, p2(75.0f / 524288.0f, -105.0f / 524288.0f), u2);
    const float2 q0 = p2(-1.0f / 64.0f, 3.0f / 64.0f), sq = p2_add(rq.h, q0);   // Q = r8 (q0 + rem)
    const df2 Q = df2_mul({p2(r8.hi, r8.hi), p2(r8.lo, r8.lo)},
                          {sq, p2_add(rq.l, p2_sub(rq.h, p2_sub(sq, q0)))});
    const df2 m = {p2(-sc.h.x, sc.h.y), p2(-sc.l.x, sc.l.y)};
    J = df2_add(cs, df2_dot2(dP, cs, Q, m));
    N = df2_add(m, df2_dot2(dP, m, {p2_neg(Q.h), p2_neg(Q.l)}, cs));
}

// ---- small arguments (x < 8) ----
// The A&S 9.1.10-9.1.11 ascending series with the logarithmic parts taken
// out, as in the FP64 routine:
//   J0 = A0,  Y0 = (2/pi) ln(x/2) J0 + A1,
//   J1 = x A2, Y1 = (2/pi) ln(x/2) J1 - 2/(pi x) + x A3,
// ten Horner terms in t = (x^2 - (4 k + 2)) / 2 on the interval k of x^2, two
// functions at a time (tables kASJY0, kASJY01 of bessel_cheb.h): the four highest terms
// (|c| <= 4e-8) in binary32, six in double-float.  About a quarter of the
// instructions of one Clenshaw sum of 17 Chebyshev terms per function.
constexpr int kASPair = 8;   // float4 per interval and pair

// (A_a, A_b) at t from the pair's eight float4
__device__ __forceinline__ df2 df2_small_series(const float4 *f, dfv t) {
    const float2 th = p2(t.hi, t.hi);
    const float4 f0 = f[0], f1 = f[1];
    float2 a = p2_fma(p2(f0.x, f0.y), th, p2(f0.z, f0.w));
    a = p2_fma(a, th, p2(f1.x, f1.y));
    a = p2_fma(a, th, p2(f1.z, f1.w));
    df2 s = {a, p2(0.f, 0.f)};
    const df2 tt = {th, p2(t.lo, t.lo)};
#pragma unroll
    for (int k = 2; k < kASPair; ++k) {
        const float4 c = f[k];
        float2 e;
        const float2 p = p2_prod(s, tt, e), ch = p2(c.x, c.y), h = p2_add(p, ch);
        s = df2_quick(h, p2_add(p2_two_sum_err(p, ch, h), p2_add(e, p2(c.z, c.w))));
    }
    return s;
}

// Interval of x^2 and t on it.
__device__ __forceinline__ int small_interval(dfv x, dfv &t) {
    const dfv v = df_mul(x, x);
    const int k = min((int)(v.hi * 0.25f), kAS_NI - 1);
    const dfv d = df_add_f(v, -(float)(4 * k + 2));
    t = df_make(0.5f * d.hi, 0.5f * d.lo);
    return k;
}

// (J0, Y0) at 0 < x < 8 from x and lnh = ln(x/2); tab: kASJY0 or a copy.
__device__ __forceinline__ df2 df2_bessel_small0(const float4 *tab, dfv x, dfv lnh) {
    dfv t;
    const int k = small_interval(x, t);
    const df2 A = df2_small_series(tab + k * kASPair, t);
    const dfv L = df_mul(df_make(kLogConstDF[2], kLogConstDF[3]), lnh);   // (2/pi) ln(x/2)
    return df2_make(df2_x(A), df_mad(L, df2_x(A), df2_y(A)));
}

// J = (J0, J1) and N = -(Y0, Y1); r8 = 8 / x; tab: kASJY01 or a copy.
__device__ __forceinline__ void df2_bessel_small01(const float4 *tab, dfv x, dfv r8, dfv lnh, df2 &J, df2 &N) {
    dfv t;
    const float4 *f = tab + 2 * kASPair * small_interval(x, t);
    const df2 A = df2_small_series(f, t), B = df2_small_series(f + kASPair, t);   // (A0, A2), (A1, A3)
    const dfv two_pi = df_make(kLogConstDF[2], kLogConstDF[3]);
    const dfv L = df_mul(two_pi, lnh);
    J = df2_make(df2_x(A), df_mul(x, df2_y(A)));
    // x A3 - 2/(pi x)
    const dfv tpx = df_mul(df_make(-0.125f * two_pi.hi, -0.125f * two_pi.lo), r8);
    const df2 b = df2_make(df2_x(B), df_mad(x, df2_y(B), tpx));
    float2 e;
    const float2 p = p2_prod(df2_bcast(L), J, e), h = p2_add(p, b.h);
    const df2 Y = df2_quick(h, p2_add(p2_two_sum_err(p, b.h, h), p2_add(e, b.l)));
    N = {p2_neg(Y.h), p2_neg(Y.l)};
}

// ln a for a double-float a > 0 (normal): a = m 2^e with m in [1/sqrt2, sqrt2),
// ln m = 2 s sum_k s^2k / (2k+1), s = (m - 1)/(m + 1), |s| <= 0.172; the
// series to k = 10 (truncation < 1e-17), terms k >= 5 (< 3e-9) in binary32.
__device__ __forceinline__ dfv df_log(dfv a) {
    int e;
    float m = frexpf(a.hi, &e);           // a.hi = m 2^e, m in [1/2, 1)
    if (m < 0.70710678f) {
        m *= 2.f;
        --e;
    }
    const dfv mm = df_make(m, ldexpf(a.lo, -e));   // exact power-of-two scaling
    const dfv s = df_mul(df_add_f(mm, -1.f), df_rcp(df_add_f(mm, 1.f)));
    const dfv s2 = df_mul(s, s);
    float pf = kAtanhDF[20];
#pragma unroll
    for (int k = 9; k >= 5; --k) pf = fmaf(pf, s2.hi, kAtanhDF[2 * k]);
    dfv p = df_make(pf, 0.f);
#pragma unroll
    for (int k = 4; k >= 0; --k) p = df_add(df_mul(p, s2), df_make(kAtanhDF[2 * k], kAtanhDF[2 * k + 1]));
    const dfv ln2 = df_make(kLogConstDF[0], kLogConstDF[1]);
    return df_add(df_mul_f(ln2, (float)e), df_mul(df_make(2.f * s.hi, 2.f * s.lo), p));
}

// Out of line: a rarely taken branch of the large kernels (its code stays out
// of the instruction stream of the common path).
static __device__ __noinline__ void df_expi_cold(double x, dfv &c, dfv &s) { df_expi(x, c, s); }

}  // namespace fh
