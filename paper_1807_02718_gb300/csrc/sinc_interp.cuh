// Interpolation of a function that is band-limited to [-pi, pi] from its
// samples at the half-integers: f(y) = sum_g f(g/2) sinc(2u) E(u), u = y - g/2,
// with the window E(u) = exp(beta (sqrt(1 - (u/U)^2) - 1)) on |u| < U = 10.5, beta =
// 32.5 (kSincU, kSincBeta): kSincPts = 42 samples, error ~1e-15 of max |f|.
// The weights are formed in double-float.
#pragma once

#include "dfloat.cuh"
#include "fh_internal.h"

namespace fh {

// e^x in double-float for -88 < x <= 0: x = k ln2 + r with |r| <= ln2 / 2,
// ln2 = L1 + L2 where L1 holds 16 significant bits (k L1 exact for |k| < 2^8);
// e^r by its Taylor series at 0, the terms n = 8 .. 13 (below 6e-9 for
// |r| <= 0.347) in binary32 and the rest in double-float; then e^x = 2^k e^r.
constexpr double kLn2 = 0.69314718055994530942;
constexpr float kLn2A = 0.693145751953125f;
constexpr float kLn2B = (float)(kLn2 - 0.693145751953125);
constexpr float kLn2C = (float)(kLn2 - 0.693145751953125 - (double)kLn2B);

// v as a double-float constant
__host__ __device__ constexpr dfv df_const(double v) { return {(float)v, (float)(v - (double)(float)v)}; }

__device__ __forceinline__ dfv df_exp(dfv x) {
    const float k = rintf(x.hi * 1.4426950408889634f);
    // r = x - k ln2: x.hi - k L1 is exact (Sterbenz), k L2 exact as a pair
    const float kb = k * kLn2B, kbe = fmaf(k, kLn2B, -kb);
    const dfv r = df_add({x.hi - k * kLn2A, x.lo}, {-kb, -fmaf(k, kLn2C, kbe)});
    float tail = 1.f / 6227020800.f;   // 1/13!
    tail = fmaf(tail, r.hi, 1.f / 479001600.f);
    tail = fmaf(tail, r.hi, 1.f / 39916800.f);
    tail = fmaf(tail, r.hi, 1.f / 3628800.f);
    tail = fmaf(tail, r.hi, 1.f / 362880.f);
    tail = fmaf(tail, r.hi, 1.f / 40320.f);
    constexpr dfv c[8] = {df_const(1.0 / 5040.0), df_const(1.0 / 720.0), df_const(1.0 / 120.0), df_const(1.0 / 24.0),
                          df_const(1.0 / 6.0), df_const(0.5), df_const(1.0), df_const(1.0)};
    dfv q = {tail, 0.f};
#pragma unroll
    for (int n = 0; n < 8; ++n) q = df_mad(q, r, c[n]);
    const int ki = (int)k;
    return {ldexpf(q.hi, ki), ldexpf(q.lo, ki)};
}

// A point y (exact in FP64) for the interpolation: the first sample row g0 =
// floor(2y) - 20, the nearest one gc, uc = y - gc/2 (|uc| <= 1/4, exact, so that
// sin(2 pi u) / u stays accurate as u -> 0) and s2 = sin(2 pi y).
struct SincPoint {
    int g0, gc;
    dfv uc, s2;
};
__device__ __forceinline__ SincPoint sinc_point(double y) {
    SincPoint p;
    p.gc = (int)rint(2.0 * y);
    p.g0 = (int)floor(2.0 * y) - (kSincPts / 2 - 1);
    p.uc = df_from(y - 0.5 * (double)p.gc);
    double sn, cs;
    sincospi(y, &sn, &cs);
    p.s2 = df_from(2.0 * sn * cs);
    return p;
}

// sinc(2u) E(u) of sample row g0 + i: sin(2 pi u) = (-1)^g sin(2 pi y), and with x =
// (u/U)^2 the exponent beta (sqrt(1 - x) - 1) = -beta x / (1 + sqrt(1 - x)), small
// where E is near 1 (as a difference it carries beta times the rounding).
__device__ __forceinline__ dfv sinc_weight(const SincPoint &p, int i) {
    const dfv u = df_add_f(p.uc, 0.5f * (float)(p.gc - p.g0 - i));
    if (u.hi == 0.f && u.lo == 0.f) return {1.f, 0.f};
    const dfv x = df_mul(df_mul(u, u), df_const(1.0 / (kSincU * kSincU)));
    const dfv w2 = df_add_f(df_neg(x), 1.f);
    if (!(w2.hi > 0.f)) return {0.f, 0.f};
    const dfv arg = df_mul(df_mul_f(x, (float)-kSincBeta), df_rcp(df_add_f(df_sqrt(w2), 1.f)));
    const dfv s2 = ((p.g0 + i) & 1) ? df_neg(p.s2) : p.s2;
    return df_mul(df_mul(s2, df_exp(arg)), df_rcp(df_mul(u, df_const(2.0 * kPi))));
}

}  // namespace fh
