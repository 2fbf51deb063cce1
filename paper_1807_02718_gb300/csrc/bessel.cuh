// J0, Y0, J1, Y1 in FP64 for x > 0, evaluated together (one sincos, one log).
//
//   x < 8:  J0 = A0, Y0 = (2/pi) ln(x/2) J0 + A1, J1 = x A2,
//           Y1 = (2/pi) ln(x/2) J1 - 2/(pi x) + x A3
//           (A0..A3 are entire in x^2: the ascending series of A&S 9.1.10-9.1.11
//            with the logarithmic parts taken out; ten Horner terms on each of 16
//            intervals of x^2, a third of the FP64 instructions of one Clenshaw
//            sum of 17 Chebyshev terms over [0, 8));
//   x >= 8: H_nu(x) = sqrt(2/(pi x)) (P_nu + i Q_nu) e^{i (x - (2 nu + 1) pi/4)},
//           P0 = B0, Q0 = (8/x) B1, P1 = B2, Q1 = (8/x) B3 as functions of
//           u = (x0/x)^2 on [8, 20] and [20, inf)  (Hankel's form, A&S 9.2.5-9.2.6).
// Each B_k is a Chebyshev series (bessel_cheb.h, made by gen_bessel_cheb.py)
// summed by Clenshaw's recurrence.  Absolute error is
// ~2e-16 for O(1) values (see the GPU test against reference tables).
#pragma once

#include "bessel_cheb.h"

namespace fh {

template <int N>
__device__ __forceinline__ double clenshaw(const double *c, double t) {
    double b1 = 0.0, b2 = 0.0;
    const double t2 = 2.0 * t;
#pragma unroll
    for (int k = N - 1; k >= 1; --k) {
        const double b0 = fma(t2, b1, c[k] - b2);
        b2 = b1;
        b1 = b0;
    }
    return fma(t, b1, c[0] - b2);
}

constexpr double kTwoOverPi = 0.63661977236758134308;
constexpr double kSqrtHalf = 0.70710678118654752440;

// Large-argument form: P0, Q0 (and P1, Q1 when want1) at x >= 8.
template <bool want1>
__device__ __forceinline__ void hankel_pq(double x, double &P0, double &Q0, double &P1,
                                          double &Q1) {
    const double r8 = 8.0 / x;
    if (x < 20.0) {
        const double u = r8 * r8;
        const double t = (u - kBLoU0) * (2.0 / (1.0 - kBLoU0)) - 1.0;
        P0 = clenshaw<kBLo0_N>(kBLo0, t);
        Q0 = r8 * clenshaw<kBLo1_N>(kBLo1, t);
        if (want1) {
            P1 = clenshaw<kBLo2_N>(kBLo2, t);
            Q1 = r8 * clenshaw<kBLo3_N>(kBLo3, t);
        }
    } else {
        const double r20 = 20.0 / x;
        const double t = 2.0 * r20 * r20 - 1.0;
        P0 = clenshaw<kBHi0_N>(kBHi0, t);
        Q0 = r8 * clenshaw<kBHi1_N>(kBHi1, t);
        if (want1) {
            P1 = clenshaw<kBHi2_N>(kBHi2, t);
            Q1 = r8 * clenshaw<kBHi3_N>(kBHi3, t);
        }
    }
}

// Horner form of P0, Q0 (and P1, Q1) for x >= 8 on 32 equal intervals of u =
// (8/x)^2, five terms each to below 1e-17 (the FP64 pipe bounds the callers, so
// short polynomials: with six intervals of x they took eight terms; fields of
// 333 targets and 200 frequencies with their synthesis 1249 -> 1120 us, FP64 kite
// of 255 systems 28.77 -> 27.93 ms, same errors).  The table
// is staged in shared memory by pq_stage() (threads of a warp may fall into
// different intervals).
struct PQShared {
    double2 c[kPU_NI * kPU_TERMS * 2];   // [interval][power of t][(P0, q0), (P1, q1)]
    double off[kPU_NI];                  // -(2 k + 1)
};

__device__ __forceinline__ void pq_stage(PQShared &tb) {
    const double2 *src = reinterpret_cast<const double2 *>(kPU);
    for (int i = threadIdx.x; i < kPU_NI * kPU_TERMS * 2; i += blockDim.x) tb.c[i] = src[i];
    for (int i = threadIdx.x; i < kPU_NI; i += blockDim.x) tb.off[i] = -(double)(2 * i + 1);
}

template <bool want1>
__device__ __forceinline__ void pq_horner(const PQShared &tb, float xf, double r8, double &P0,
                                          double &Q0, double &P1, double &Q1) {
    // (the interval in binary32: off by one at its ends is as good)
    const int k = min((int)__fdividef(64.f * kPU_NI, xf * xf), kPU_NI - 1);
    const double t = fma(r8 * r8, 2.0 * kPU_NI, tb.off[k]);
    const double2 *c = tb.c + k * kPU_TERMS * 2;
    double2 a = c[2 * (kPU_TERMS - 1)], b = want1 ? c[2 * (kPU_TERMS - 1) + 1] : make_double2(0.0, 0.0);
#pragma unroll
    for (int p = kPU_TERMS - 2; p >= 0; --p) {
        const double2 v = c[2 * p];
        a.x = fma(a.x, t, v.x);
        a.y = fma(a.y, t, v.y);
        if (want1) {
            const double2 w = c[2 * p + 1];
            b.x = fma(b.x, t, w.x);
            b.y = fma(b.y, t, w.y);
        }
    }
    P0 = a.x;
    Q0 = r8 * a.y;
    if (want1) {
        P1 = b.x;
        Q1 = r8 * b.y;
    }
}

// A0..A3 at x < 8 (the first kF of them; order A0, A1, A2, A3), tab = kAS or a
// copy of it in shared memory.
template <int kF>
__device__ __forceinline__ void small_series(const double *tab, double x, double (&a)[kF]) {
    const double v = x * x;
    const int k = min((int)((float)v * 0.25f), kAS_NI - 1);
    const double t = fma(v, 0.5, -(double)(2 * k + 1));
    const double *c = tab + k * 4 * kAS_TERMS;
#pragma unroll
    for (int f = 0; f < kF; ++f) {
        double s = c[f * kAS_TERMS + kAS_TERMS - 1];
#pragma unroll
        for (int p = kAS_TERMS - 2; p >= 0; --p) s = fma(s, t, c[f * kAS_TERMS + p]);
        a[f] = s;
    }
}

// Small-argument branch (x < 8) with lnh = ln(x/2) and r8 = 8/x given (both
// shared by a frequency group).
__device__ __forceinline__ void bessel_small_ln(const double *tab, double x, double r8, double lnh, double &J0,
                                                double &Y0, double &J1, double &Y1) {
    double a[4];
    small_series(tab, x, a);
    const double L = kTwoOverPi * lnh;
    J0 = a[0];
    Y0 = fma(L, J0, a[1]);
    J1 = x * a[2];
    Y1 = fma(L, J1, fma(x, a[3], -0.125 * kTwoOverPi * r8));
}

__device__ __forceinline__ void bessel_small0_ln(const double *tab, double x, double lnh, double &J0, double &Y0) {
    double a[2];
    small_series(tab, x, a);
    J0 = a[0];
    Y0 = fma(kTwoOverPi * lnh, J0, a[1]);
}

__device__ __forceinline__ void bessel_j0y0j1y1(double x, double &J0, double &Y0, double &J1,
                                                double &Y1) {
    if (x < 8.0) {
        bessel_small_ln(kAS, x, 8.0 / x, log(0.5 * x), J0, Y0, J1, Y1);
    } else {
        double s, c;
        sincos(x, &s, &c);
        const double c0 = (c + s) * kSqrtHalf;   // cos(x - pi/4)
        const double s0 = (s - c) * kSqrtHalf;   // sin(x - pi/4)
        double P0, Q0, P1, Q1;
        hankel_pq<true>(x, P0, Q0, P1, Q1);
        const double A = sqrt(kTwoOverPi / x);
        J0 = A * (P0 * c0 - Q0 * s0);
        Y0 = A * (P0 * s0 + Q0 * c0);
        J1 = A * (P1 * s0 + Q1 * c0);   // chi_1 = chi_0 - pi/2
        Y1 = A * (Q1 * s0 - P1 * c0);
    }
}

__device__ __forceinline__ void bessel_j0y0(double x, double &J0, double &Y0) {
    if (x < 8.0) {
        bessel_small0_ln(kAS, x, log(0.5 * x), J0, Y0);
    } else {
        double s, c;
        sincos(x, &s, &c);
        const double c0 = (c + s) * kSqrtHalf, s0 = (s - c) * kSqrtHalf;
        double P0, Q0, P1, Q1;
        hankel_pq<false>(x, P0, Q0, P1, Q1);
        const double A = sqrt(kTwoOverPi / x);
        J0 = A * (P0 * c0 - Q0 * s0);
        Y0 = A * (P0 * s0 + Q0 * c0);
    }
}

}  // namespace fh
