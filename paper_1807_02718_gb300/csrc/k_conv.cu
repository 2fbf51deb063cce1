// The FFT-accelerated scaled convolution (Sec. 4.1.2).
//
// d_n = sum_m c_m b(beta n - gamma m) (eqs. conv_sum, conv_sum_2 with the
// index reading of eq. discConv) is approximated by eq. approx_conv_sum:
// C^{(gamma)}_p (gamma-fractional DFT of c zero-padded to L), B_p (DFT of b at
// the integers -L/2..L/2-1) and the inverse beta-fractional DFT of C B.
//
// A fractional DFT of length L is computed by the chirp factorisation 2mp =
// m^2 + p^2 - (p - m)^2 as one circular convolution of length Nf >= 2L (a
// power of two) with the filter e^{i pi alpha k^2 / L}; a DFT (alpha = 1) of a
// power-of-two length is one FFT.
//
// FFT.  The work is bound by the FP64 pipe (1/64 of the FP32 rate: about 3.5
// FP64 instructions per element and factor of two in radix 8 with tabulated
// roots, against 16 bytes per element and pass that stay in L2), so the
// kernels keep the instruction count and the number of passes down:
//  - a line of 2^A <= 4096 points is transformed inside one CTA, eight points
//    per thread in registers, radix-8 Stockham passes exchanged through
//    shared memory, every root read from a table (no sincos);
//  - a row of Nf = N1 N2 points is N2 columns of N1 points (element i = i1 N2
//    + i2), the roots w^{i2 k1}, then N1 lines of N2 points, which leaves
//    X[k1 + N1 k2] at k1 N2 + k2.  A convolution multiplies two transforms in
//    that order and goes back the same way, so nothing is ever transposed and
//    it takes three launches: columns forward (the chirp and the zero padding
//    applied while loading), lines forward + filter + lines backward, columns
//    backward (the chirp, the middle factor and the scale while storing);
//  - the chirps e^{i pi alpha k^2 / L} are tabulated once per alpha and serve
//    the loads, the stores and the filter; at gamma = 1 both transforms of c
//    and of b use one filter.
// Measured (GB300; out-of-place radix-2 stages with a sincospi per butterfly
// before): 64 traces of L = 16384, M = 1000: 7.38 -> 0.71 ms; one trace of L =
// 10^6, M = 5000: 20.2 -> 3.12 ms (eight FFTs of 2^21 points, 1.2e9 FP64
// instructions: 2.3 ms where a warp's addition or product holds the pipe for 19
// clocks, as measured; an FMA holds it for 16).
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "fh_internal.h"
#include "scratch.cuh"

namespace fh {
namespace {

constexpr int kRootBits = 12, kRoots = 1 << kRootBits;   // roots of unity of order 4096
constexpr int kLine = 4096;                              // points of the longest line
constexpr double kSqrtHalf = 0.70710678118654752440;

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 conj2(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double2 add2(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 sub2(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }

// v mod 2 in (-1, 1], exactly: the nearest even integer is subtracted by an FMA
__device__ __forceinline__ double mod2(double v) { return fma(-2.0, rint(0.5 * v), v); }

// (a N / D) mod 2 for integers N, D > 0: N = q D + r exactly, a q as an
// exact two-term product, reduced modulo 2 before the small terms are added,
// so that the phase pi a N / D keeps its accuracy for large N.
__device__ __forceinline__ double mulmod2(double a, long long N, long long D) {
    long long q = N / D, r = N - q * D;
    if (r < 0) {
        r += D;
        --q;
    }
    const double hi = a * (double)q;
    const double lo = fma(a, (double)q, -hi);
    return mod2(mod2(hi) + lo + a * (double)r / (double)D);
}

__device__ __forceinline__ double2 expi_pi(double r) {   // e^{i pi r}
    double s, c;
    sincospi(r, &s, &c);
    return make_double2(c, s);
}

// chirp[k] = e^{i pi alpha k^2 / L}, 0 <= k < L.  The quotient of k^2 by L
// comes from a binary64 product (k^2 < 2^48 and its quotient are exact
// integers), corrected by one.
__global__ void chirp_table_kernel(int L, double alpha, double inv_L, double2 *__restrict__ chirp) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= L) return;
    const long long kk = (long long)k * k;
    long long q = (long long)((double)kk * inv_L);
    long long r = kk - q * L;
    if (r < 0) {
        r += L;
        --q;
    } else if (r >= L) {
        r -= L;
        ++q;
    }
    const double hi = alpha * (double)q;
    const double lo = fma(alpha, (double)q, -hi);
    chirp[k] = expi_pi(mod2(mod2(hi) + lo + alpha * (double)r * inv_L));
}

// roots[j] = e^{-2 pi i j / 4096}; fine[j] = e^{-2 pi i j / Nf}, j < 4096: w_Nf^e =
// roots[(e >> 12) 4096^2 / Nf] fine[e & 4095].
__global__ void roots_kernel(double nf, double2 *__restrict__ roots, double2 *__restrict__ fine) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= kRoots) return;
    roots[j] = expi_pi(-2.0 * (double)j / (double)kRoots);
    fine[j] = expi_pi(-2.0 * (double)j / nf);
}

__device__ __forceinline__ double2 root_nf(const double2 *__restrict__ roots, const double2 *__restrict__ fine,
                                           int bits, int e) {   // w_Nf^e, Nf = 2^bits > 4096, e < Nf
    return cmul(__ldg(roots + ((e >> kRootBits) << (2 * kRootBits - bits))), __ldg(fine + (e & (kRoots - 1))));
}

// ---- one line of n = 2^A points: eight per thread, n / 8 threads ----
// Thread t holds the points t + q n/8, q < 8, before the first and after the
// last pass.  Pass with radix R after passes of product Ls (Stockham): the
// butterflies j = t + i n/8 (i < 8/R) take the points j + r n/R = t + (i + r
// 8/R) n/8, multiply by w_{Ls R}^{k r} (k = j mod Ls), and put output r at
// (j / Ls) Ls R + k + r Ls.

template <int S> __device__ __forceinline__ double2 rot(double2 a) {   // a * (S i)
    return S < 0 ? make_double2(a.y, -a.x) : make_double2(-a.y, a.x);
}

template <int S> __device__ __forceinline__ void dft4(double2 &a, double2 &b, double2 &c, double2 &d) {
    const double2 t0 = add2(a, c), t1 = sub2(a, c), t2 = add2(b, d), t3 = rot<S>(sub2(b, d));
    a = add2(t0, t2);
    b = add2(t1, t3);
    c = sub2(t0, t2);
    d = sub2(t1, t3);
}

template <int S> __device__ __forceinline__ void dft8(double2 (&v)[8]) {
    double2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4<S>(e0, e1, e2, e3);
    dft4<S>(o0, o1, o2, o3);
    constexpr double s = (double)S;
    o1 = make_double2(kSqrtHalf * (o1.x - s * o1.y), kSqrtHalf * (o1.y + s * o1.x));
    o2 = rot<S>(o2);
    o3 = make_double2(-kSqrtHalf * (o3.x + s * o3.y), kSqrtHalf * (s * o3.x - o3.y));
    v[0] = add2(e0, o0); v[4] = sub2(e0, o0);
    v[1] = add2(e1, o1); v[5] = sub2(e1, o1);
    v[2] = add2(e2, o2); v[6] = sub2(e2, o2);
    v[3] = add2(e3, o3); v[7] = sub2(e3, o3);
}

__device__ __forceinline__ int pad8(int i) { return i + (i >> 3); }   // conflict-free strides of 8 points

template <int A, int R, int Ls, int S, bool kLast>
__device__ __forceinline__ void fft_pass(double2 (&v)[8], int t, double2 *line, const double2 *__restrict__ roots) {
    constexpr int n = 1 << A, E = n / 8, G = 8 / R;
#pragma unroll
    for (int i = 0; i < G; ++i) {
        const int k = (t + i * E) & (Ls - 1);
        if (Ls > 1) {
#pragma unroll
            for (int r = 1; r < R; ++r) {
                double2 w = __ldg(roots + k * r * (kRoots / (Ls * R)));
                if (S > 0) w.y = -w.y;
                v[i + r * G] = cmul(v[i + r * G], w);
            }
        }
    }
    if constexpr (R == 8) {
        dft8<S>(v);
    } else if constexpr (R == 4) {
#pragma unroll
        for (int i = 0; i < G; ++i) dft4<S>(v[i], v[i + G], v[i + 2 * G], v[i + 3 * G]);
    } else {
#pragma unroll
        for (int i = 0; i < G; ++i) {
            const double2 a = v[i], b = v[i + G];
            v[i] = add2(a, b);
            v[i + G] = sub2(a, b);
        }
    }
    if constexpr (!kLast) {
        __syncthreads();   // the points of the pass before are read
#pragma unroll
        for (int i = 0; i < G; ++i) {
            const int j = t + i * E, k = j & (Ls - 1), o = (j - k) * R + k;
#pragma unroll
            for (int r = 0; r < R; ++r) line[pad8(o + r * Ls)] = v[i + r * G];
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = line[pad8(t + q * E)];
    }
}

// Forward (S = -1): the remainder radix 2^(A mod 3) first, then radix 8, so
// that the last pass leaves each thread the points with which the radix-8
// pass of the backward transform (S = 1: radix 8 first, the remainder last)
// begins; both are in natural order on both sides.
template <int A, int Ls, int S>
__device__ __forceinline__ void fft_passes(double2 (&v)[8], int t, double2 *line, const double2 *__restrict__ roots) {
    constexpr int n = 1 << A, left = n / Ls, rem = 1 << (A % 3);
    constexpr int R = S < 0 ? ((Ls == 1 && rem > 1) ? rem : 8) : (left >= 8 ? 8 : left);
    fft_pass<A, R, Ls, S, (Ls * R == n)>(v, t, line, roots);
    if constexpr (Ls * R < n) fft_passes<A, Ls * R, S>(v, t, line, roots);
}
template <int A, int S>
__device__ __forceinline__ void fft_line(double2 (&v)[8], int t, double2 *line, const double2 *__restrict__ roots) {
    static_assert(A >= 3 && A <= 12, "a line has 8 to 4096 points");
    fft_passes<A, 1, S>(v, t, line, roots);
}

__host__ __device__ constexpr int line_stride(int n) { return n + n / 8 + 2; }   // shared memory of a line

// ---- what the first pass reads and the last one writes ----

// Row b, point i < Nf of a transform's input.
struct Source {
    enum Kind { kPadded, kRows, kKernel, kFilter, kRaw } kind;
    const double2 *src = nullptr;      // kPadded: batch x M rows about L/2; kRows: batch x L; kRaw: batch x nf
    const double2 *chirp = nullptr;    // multiplied by its conjugate at |i - L/2|; null: by (-1)^i (plain DFT)
    int L = 0, M = 0, nf = 0;
    double A = 0.0, r = 0.0;           // kKernel: b(q) = 2A sinc(r q), r = 2A / P

    __device__ __forceinline__ double2 at(long long b, int i) const {
        if (kind == kRaw) return src[b * nf + i];
        double2 v = make_double2(0.0, 0.0);
        if (kind == kFilter) {         // chirp at k and Nf - k, |k| < L
            if (i < L) v = __ldg(chirp + i);
            else if (i > nf - L) v = __ldg(chirp + (nf - i));
            return v;
        }
        if (i >= L) return v;
        const int m = i - L / 2;
        if (kind == kPadded) {
            if (m < -(M / 2) || m >= M / 2) return v;
            v = src[b * M + (m + M / 2)];
        } else if (kind == kRows) {
            v = src[b * L + i];
        } else {
            const double y = r * (double)m;
            v.x = 2.0 * A * (m == 0 ? 1.0 : sinpi(y) / (kPi * y));
        }
        if (chirp) return cmul(v, conj2(__ldg(chirp + (m < 0 ? -m : m))));
        return (i & 1) ? make_double2(-v.x, -v.y) : v;
    }
};

// Row b, point i of a transform's output (points i >= L are dropped).
struct Sink {
    double2 *dst = nullptr;            // batch x L
    const double2 *chirp = nullptr;    // as in Source (plain DFT: (-1)^(i + L/2))
    const double2 *mid = nullptr;      // multiplied by mid[i] (may be null)
    int L = 0;
    double beta = 0.0;                 // with_phase: multiplied by e^{2 pi i beta n0 p / L}, p = i - L/2
    long long n0 = 0;
    bool with_phase = false;
    int raw_nf = 0;                    // > 0: the points themselves, batch x raw_nf

    __device__ __forceinline__ void put(long long b, int i, double2 v) const {
        if (raw_nf) {
            dst[b * raw_nf + i] = v;
            return;
        }
        if (i >= L) return;
        const int p = i - L / 2;
        if (chirp) v = cmul(v, conj2(__ldg(chirp + (p < 0 ? -p : p))));
        else if (p & 1) v = make_double2(-v.x, -v.y);
        if (mid) v = cmul(v, __ldg(mid + i));
        if (with_phase) {
            const long long np = n0 * p;
            const double ph = np >= 0 ? mulmod2(2.0 * beta, np, L) : -mulmod2(2.0 * beta, -np, L);
            v = cmul(v, expi_pi(ph));
        }
        dst[b * L + i] = v;
    }
};

// Columns of n = 2^A = N1 points, c adjacent ones per CTA (contiguous loads of
// c points; thread order column-fastest).
__host__ __device__ constexpr int columns_per_cta(int A) { return A <= 9 ? 8 : kLine >> A; }

template <int A, bool kForward>
__global__ void __launch_bounds__((1 << A) / 8 * columns_per_cta(A)) fft_columns_kernel(
    int bits, Source in, Sink out, double2 *Y, const double2 *__restrict__ roots,
    const double2 *__restrict__ fine) {
    constexpr int n = 1 << A, c = columns_per_cta(A), E = n / 8;
    extern __shared__ double2 sm[];
    const int N2 = 1 << (bits - A);
    const int line = threadIdx.x % c, t = threadIdx.x / c;
    const long long groups = N2 / c, b = blockIdx.x / groups;
    const int i2 = (int)(blockIdx.x % groups) * c + line;
    double2 *row = Y + (b << bits);
    double2 v[8];
    if (kForward) {
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = in.at(b, (t + q * E) * N2 + i2);
        fft_line<A, -1>(v, t, sm + line * line_stride(n), roots);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int k1 = t + q * E;
            row[(long long)k1 * N2 + i2] = cmul(v[q], root_nf(roots, fine, bits, k1 * i2));
        }
    } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = row[(long long)(t + q * E) * N2 + i2];
        fft_line<A, 1>(v, t, sm + line * line_stride(n), roots);
#pragma unroll
        for (int q = 0; q < 8; ++q) out.put(b, (t + q * E) * N2 + i2, v[q]);
    }
}

// Lines of n = 2^A = N2 points (N1 = 2^(bits - A) of them per row).
//   kMode 0: Y = scale * transform, in the order of the lines (a filter)
//   kMode 1: forward, times the filter Z (row b mod z_rows), backward (the
//            roots w^{-i2 k1} on the way out)
//   kMode 2: forward, to the sink at k1 + N1 k2 (plain DFT)
// N1 = 1: the source is read and the sink written here (no column pass).
__host__ __device__ constexpr int lines_per_cta(int A) { return A >= 9 ? 1 : 512 >> A; }

template <int A, int kMode>
__global__ void __launch_bounds__((1 << A) / 8 * lines_per_cta(A)) fft_lines_kernel(
    int bits, long long batch, Source in, Sink out, double2 *Y, const double2 *Z, int z_rows, double scale,
    const double2 *__restrict__ roots, const double2 *__restrict__ fine) {
    constexpr int n = 1 << A, E = n / 8;
    extern __shared__ double2 sm[];
    const int N1 = 1 << (bits - A);
    const int ln = threadIdx.x / E, t = threadIdx.x % E;
    const long long g = (long long)blockIdx.x * lines_per_cta(A) + ln;   // line of the batch
    const bool valid = g < batch * N1;
    const long long b = g >> (bits - A);
    const int k1 = (int)(g & (N1 - 1));
    double2 *lineY = Y + (b << bits) + (long long)k1 * n;
    double2 v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int i = t + q * E;
        v[q] = !valid ? make_double2(0.0, 0.0) : N1 == 1 ? in.at(b, i) : lineY[i];
    }
    double2 *line = sm + ln * line_stride(n);
    fft_line<A, -1>(v, t, line, roots);
    if (kMode == 0) {
        if (valid)
#pragma unroll
            for (int q = 0; q < 8; ++q)
                lineY[t + q * E] = make_double2(scale * v[q].x, scale * v[q].y);
        return;
    }
    if (kMode == 2) {
        if (valid)
#pragma unroll
            for (int q = 0; q < 8; ++q) out.put(b, k1 + (t + q * E) * N1, v[q]);
        return;
    }
    const double2 *z = Z + ((b & (z_rows - 1)) << bits) + (long long)k1 * n;
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = cmul(v[q], __ldg(z + t + q * E));
    fft_line<A, 1>(v, t, line, roots);
    if (!valid) return;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int i = t + q * E;
        if (N1 == 1) out.put(b, i, v[q]);
        else lineY[i] = cmul(v[q], conj2(root_nf(roots, fine, bits, k1 * i)));
    }
}

// Rows of 2^25 points (L > 2^23): one radix-2 step splits a row into the two
// half rows 2b (even outputs) and 2b + 1 (odd outputs), and joins them again;
// the launches above then see rows of 2^24.
__global__ void split_rows_kernel(int half_bits, long long batch, Source in, double2 *__restrict__ Y) {
    const int h = 1 << half_bits, i = blockIdx.x * blockDim.x + threadIdx.x;
    const long long b = blockIdx.y;
    if (i >= h) return;
    const double2 x0 = in.at(b, i), x1 = in.at(b, i + h);
    Y[((2 * b) << half_bits) + i] = add2(x0, x1);
    Y[((2 * b + 1) << half_bits) + i] = cmul(sub2(x0, x1), expi_pi(-(double)i / (double)h));
}
__global__ void join_rows_kernel(int half_bits, long long batch, const double2 *__restrict__ Y, Sink out) {
    const int h = 1 << half_bits, i = blockIdx.x * blockDim.x + threadIdx.x;
    const long long b = blockIdx.y;
    if (i >= h) return;   // L <= 2^24 = h: the second half of the row is not needed
    const double2 u0 = Y[((2 * b) << half_bits) + i], u1 = Y[((2 * b + 1) << half_bits) + i];
    out.put(b, i, add2(u0, cmul(u1, expi_pi((double)i / (double)h))));
}

// ---- host helpers ----

unsigned grid_of(long long n, int block) { return (unsigned)((n + block - 1) / block); }

struct Fft {
    cudaStream_t st;
    const double2 *roots, *fine;   // of the row length in question
    int bits;                      // row length 2^bits

    // Bits of N1: none up to one line; else about half of them, where columns
    // are loaded four or eight at a time (64 bytes or more), and whatever a
    // line of 4096 leaves.
    int column_bits() const {
        if (bits <= 12) return 0;
        return std::max(std::min(bits / 2, 10), bits - 12);
    }
    template <bool kForward>
    void columns(long long rows, const Source &in, const Sink &out, double2 *Y) const {
        const int a = column_bits();
        auto go = [&](auto a_c) {
            constexpr int A = decltype(a_c)::value;
            constexpr int c = columns_per_cta(A), smem = c * line_stride(1 << A) * (int)sizeof(double2);
            static std::atomic<unsigned long long> attr{0};
            ensure_smem_attr((const void *)fft_columns_kernel<A, kForward>, smem, attr);
            const long long ctas = rows * ((1ll << (bits - A)) / c);
            fft_columns_kernel<A, kForward><<<(unsigned)ctas, (1 << A) / 8 * c, smem, st>>>(bits, in, out, Y, roots, fine);
        };
        switch (a) {
            case 6: go(std::integral_constant<int, 6>{}); break;
            case 7: go(std::integral_constant<int, 7>{}); break;
            case 8: go(std::integral_constant<int, 8>{}); break;
            case 9: go(std::integral_constant<int, 9>{}); break;
            case 10: go(std::integral_constant<int, 10>{}); break;
            case 11: go(std::integral_constant<int, 11>{}); break;
            case 12: go(std::integral_constant<int, 12>{}); break;
        }
    }
    template <int kMode>
    void lines(long long rows, const Source &in, const Sink &out, double2 *Y, const double2 *Z, int z_rows,
               double scale) const {
        auto go = [&](auto a_c) {
            constexpr int A = decltype(a_c)::value;
            constexpr int l = lines_per_cta(A), smem = l * line_stride(1 << A) * (int)sizeof(double2);
            static std::atomic<unsigned long long> attr{0};
            ensure_smem_attr((const void *)fft_lines_kernel<A, kMode>, smem, attr);
            const long long n_lines = rows << (bits - A);
            fft_lines_kernel<A, kMode><<<grid_of(n_lines, l), (1 << A) / 8 * l, smem, st>>>(
                bits, rows, in, out, Y, Z, z_rows, scale, roots, fine);
        };
        switch (bits - column_bits()) {
            case 3: go(std::integral_constant<int, 3>{}); break;
            case 4: go(std::integral_constant<int, 4>{}); break;
            case 5: go(std::integral_constant<int, 5>{}); break;
            case 6: go(std::integral_constant<int, 6>{}); break;
            case 7: go(std::integral_constant<int, 7>{}); break;
            case 8: go(std::integral_constant<int, 8>{}); break;
            case 9: go(std::integral_constant<int, 9>{}); break;
            case 10: go(std::integral_constant<int, 10>{}); break;
            case 11: go(std::integral_constant<int, 11>{}); break;
            case 12: go(std::integral_constant<int, 12>{}); break;
        }
    }
    static Source raw_source(const double2 *Y, int nf) {
        Source s{Source::kRaw};
        s.src = Y;
        s.nf = nf;
        return s;
    }
    static Sink raw_sink(double2 *Y, int nf) {
        Sink s;
        s.dst = Y;
        s.raw_nf = nf;
        return s;
    }
    // rows of 2^25 points as twice as many of 2^24
    Fft half() const { return Fft{st, roots, fine, bits - 1}; }

    // The filter Y = scale * FFT(in), one row, in the order of the lines.
    void filter(const Source &in, double2 *Y, double scale) const {
        if (bits > 24) {
            split_rows_kernel<<<dim3(1u << (bits - 1 - 8), 1), 256, 0, st>>>(bits - 1, 1, in, Y);
            const Fft f = half();
            f.columns<true>(2, raw_source(Y, 1 << f.bits), Sink{}, Y);
            f.lines<0>(2, Source{Source::kRaw}, Sink{}, Y, nullptr, 1, scale);
            return;
        }
        if (column_bits()) columns<true>(1, in, Sink{}, Y);
        lines<0>(1, in, Sink{}, Y, nullptr, 1, scale);
    }
    // out = FFT^-1(FFT(in) Z) for `rows` rows (Y: work space, rows << bits points).
    void convolve(long long rows, const Source &in, const Sink &out, double2 *Y, const double2 *Z) const {
        if (bits > 24) {
            split_rows_kernel<<<dim3(1u << (bits - 1 - 8), (unsigned)rows), 256, 0, st>>>(bits - 1, rows, in, Y);
            const Fft f = half();
            const int h = 1 << f.bits;
            f.columns<true>(2 * rows, raw_source(Y, h), Sink{}, Y);
            f.lines<1>(2 * rows, Source{Source::kRaw}, Sink{}, Y, Z, 2, 1.0);
            f.columns<false>(2 * rows, Source{Source::kRaw}, raw_sink(Y, h), Y);
            join_rows_kernel<<<dim3(1u << (bits - 1 - 8), (unsigned)rows), 256, 0, st>>>(bits - 1, rows, Y, out);
            return;
        }
        if (column_bits()) columns<true>(rows, in, Sink{}, Y);
        lines<1>(rows, in, out, Y, Z, 1, 1.0);
        if (column_bits()) columns<false>(rows, in, out, Y);
    }
    // out = DFT(in) of length 2^bits, centred indices (the signs are in Source and Sink).
    void dft(long long rows, const Source &in, const Sink &out, double2 *Y) const {
        if (column_bits()) columns<true>(rows, in, Sink{}, Y);
        lines<2>(rows, in, out, Y, nullptr, 1, 1.0);
    }
};

}  // namespace
}  // namespace fh

using namespace fh;

extern "C" fh_status fh_scaled_convolution(const double *d_c, int M, int batch, double beta, double gamma,
                                           long long n0, int L, double A, double P, double *d_d, void *stream) {
    if (M < 2 || (M & 1) || batch < 1 || L < M || (L & 1) || !(A > 0.0) || !(P > 0.0) || !d_c || !d_d ||
        !std::isfinite(beta) || !std::isfinite(gamma) || L > (1 << 24))
        return FH_EINVAL;
    if (cudaPeekAtLastError() != cudaSuccess) return FH_ECUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int bits = 3, lbits = 3;   // a line has at least 8 points
    while ((1ll << bits) < 2ll * L) ++bits;
    while ((1ll << lbits) < L) ++lbits;
    // alpha = 1 on a power-of-two length is an ordinary DFT: one FFT of L points
    // in place of two of Nf >= 2L and a filter
    const bool plain = (1 << lbits) == L;
    const bool plain_c = plain && gamma == 1.0, chirp_1 = !plain, chirp_g = gamma != 1.0;
    const size_t nf = (size_t)1 << bits;
    fh_status status = FH_OK;
    {
        Scratch sc{{}, st};
        double2 *Y = sc.get<double2>(nf * batch);
        double2 *Z = sc.get<double2>(nf);
        double2 *Cg = sc.get<double2>((size_t)L * batch);
        double2 *Bm = sc.get<double2>((size_t)L);
        double2 *chirp = sc.get<double2>((size_t)L);
        double2 *roots = sc.get<double2>(3 * (size_t)kRoots);
        if (!Y || !Z || !Cg || !Bm || !chirp || !roots) {
            cudaGetLastError();
            return FH_ENOMEM;
        }
        // the rows of 2^25 points are transformed as rows of 2^24
        const int row_bits = std::min(bits, 24);
        roots_kernel<<<kRoots / 256, 256, 0, st>>>((double)(1 << row_bits), roots, roots + kRoots);
        if (plain) roots_kernel<<<kRoots / 256, 256, 0, st>>>((double)L, roots, roots + 2 * kRoots);
        const Fft f{st, roots, roots + kRoots, bits}, fl{st, roots, roots + 2 * kRoots, lbits};
        const double inv_nf = 1.0 / (double)nf;
        auto chirp_filter = [&](double alpha, double scale) {
            chirp_table_kernel<<<grid_of(L, 256), 256, 0, st>>>(L, alpha, 1.0 / (double)L, chirp);
            Source z{Source::kFilter};
            z.chirp = chirp;
            z.L = L;
            z.nf = (int)nf;
            f.filter(z, Z, scale);
        };
        // B_p: DFT of b at the integers, times e^{2 pi i beta n0 p / L}
        Source bsrc{Source::kKernel};
        bsrc.L = L;
        bsrc.A = A;
        bsrc.r = 2.0 * A / P;
        Sink bdst;
        bdst.dst = Bm;
        bdst.L = L;
        bdst.beta = beta;
        bdst.n0 = n0;
        bdst.with_phase = true;
        if (chirp_1) {
            chirp_filter(1.0, inv_nf);
            bsrc.chirp = bdst.chirp = chirp;
            f.convolve(1, bsrc, bdst, Y, Z);
        } else {
            fl.dft(1, bsrc, bdst, Y);
        }
        // C^{(gamma)}_p, times B_p e^{2 pi i beta n0 p / L}
        Source csrc{Source::kPadded};
        csrc.src = reinterpret_cast<const double2 *>(d_c);
        csrc.L = L;
        csrc.M = M;
        Sink cdst;
        cdst.dst = Cg;
        cdst.L = L;
        cdst.mid = Bm;
        if (plain_c) {
            fl.dft(batch, csrc, cdst, Y);
        } else {
            if (chirp_g) chirp_filter(gamma, inv_nf);
            csrc.chirp = cdst.chirp = chirp;
            f.convolve(batch, csrc, cdst, Y, Z);
        }
        // the inverse beta-fractional transform: d_{n0+n'} = (1/L) sum_p (...) e^{2 pi i beta n' p / L}
        chirp_filter(-beta, inv_nf / (double)L);
        Source dsrc{Source::kRows};
        dsrc.src = Cg;
        dsrc.chirp = chirp;
        dsrc.L = L;
        Sink ddst;
        ddst.dst = reinterpret_cast<double2 *>(d_d);
        ddst.chirp = chirp;
        ddst.L = L;
        f.convolve(batch, dsrc, ddst, Y, Z);
        if (cudaGetLastError() != cudaSuccess) status = FH_ECUDA;
    }
    return status;
}
