// Step a5 (step F5): target fields from the resident densities
//
//   V(x, omega_j) = int_Gamma psi_p(r', omega_j) G_omega(x, r') dsigma(r')
//                 ~ (pi/n) sum_i (i/4) H0(kappa |x - z_i|) |z'_i| psi_i
// (Sec. 2.3 eq. freq_domain_repr, Sec. 3.2 eq. Ukslow_repr; trapezoidal rule
// on the Nystrom nodes).  omega = 0 has no solve; V(x, 0) := 1 there (the 2D
// low-frequency limit of the radiating field with data e^{i kappa p.r}).
//
// One CTA per (frequency subgroup, chunk of nodes, tile of targets); source
// nodes are staged through shared memory with the weights (pi/n) |z'_i| psi_i /
// 4 premultiplied.
#include "bessel.cuh"
#include "dfloat.cuh"
#include "fh_internal.h"

namespace fh {
namespace {

constexpr int kTgt = 128;
constexpr int kChunk = kFieldChunk;   // largest number of source nodes per work item

// Work item w = (subgroup g, chunk of `chunk` <= kChunk nodes).  One CTA per
// (kTileF64 targets, item); thread (target tid % kTileF64, slice tid /
// kTileF64) takes every kSlicesF64-th node of the chunk, and the slices' sums are
// added in slice order (the split is the same for every n_x, so that a
// target's field does not depend on the other targets of the call).
// For each target-node pair the distance r, 1/r, the phase e^{i(kappa_0 r -
// pi/4)} with the amplitude sqrt(2/(pi r)) and the step e^{i dkappa r} are formed
// once; each frequency j of the subgroup then needs only the Horner P0/Q0
// series (x = kappa_j r >= 8) or the small-argument series (x < 8); 1 /
// sqrt(kappa_j) is on the staged densities.  The phase carries the exact
// kappa_j through a first-order correction e^{i (kappa_j - kappa_0 - j dkappa)
// r}.  Partial sums per item go to scratch; field_reduce_kernel adds them in a
// fixed order (the result does not depend on scheduling).
// Bound by the FP64 pipe: 2 FMAs per clock and SM, a warp instruction holding it
// for 16 clocks whatever its number of active lanes.  With one target per
// thread and 128 targets per CTA, 16 targets left 7 of 8 lanes idle and a CTA
// (64 nodes x 8 frequencies) held an SM for a millisecond, so that a few
// hundred targets made less than three waves of them.  Measured (GB300): 16
// targets x 63 frequencies, N = 256: 2.60 -> 0.20 ms; 1024 x 255, N 64..480:
// 8.44 -> 4.96 ms (FP64 pipe active 90 % of the cycles); spectra, fields and synthesis at 333 targets x 1001 times,
// 200 frequencies: 4.77 -> 1.9 ms (1.12 ms with the contraction's and the
// Hankel polynomials' later changes).
constexpr int kTileF64 = 16, kSlicesF64 = kTgt / kTileF64;

__global__ void __launch_bounds__(kTgt) field_partial_kernel(
    SolveTables t, Subgroups grp, const int2 *__restrict__ items, int item_begin, int chunk,
    const double2 *__restrict__ z, const double2 *__restrict__ dz,
    const double2 *__restrict__ psi, const double *__restrict__ x, int n_x,
    double2 *__restrict__ part) {
    const int w = blockIdx.y;
    const int2 item = items[item_begin + w];    // (subgroup, first node)
    const int g = item.x, i0 = item.y;
    const int2 sgv = grp.sg[g];
    const int s0 = sgv.x, cnt = sgv.y;
    const int N = t.N[s0];
    const int vo0 = t.vec_off[s0];
    const double wq = 2.0 * kPi / (double)N * 0.25;   // (pi/n) / 4
    const double dk = grp.dkappa[g];
    __shared__ double kap[kGroup], ikap8[kGroup], isqk[kGroup], sqk[kGroup], lnk2[kGroup], corr[kGroup];
    __shared__ float kapf[kGroup];
    __shared__ double2 zs[kChunk];
    __shared__ double2 ps[kGroup][kChunk];   // (pi/n)|z'|/4 * psi_j / sqrt(kappa_j) at each node
    __shared__ double2 sums[kGroup][kTgt];
    __shared__ PQShared pqt;
    pq_stage(pqt);
    if (threadIdx.x < kGroup) {
        const int j = threadIdx.x;
        const double k = (j < cnt) ? t.kappa[s0 + j] : 1.0;
        kap[j] = k;
        kapf[j] = (float)k;
        ikap8[j] = 8.0 / k;
        sqk[j] = sqrt(k);
        isqk[j] = 1.0 / sqrt(k);
        lnk2[j] = log(0.5 * k);   // ln(x/2) = ln(kappa/2) + ln r
    }
    __syncthreads();
    const int ne = min(chunk, N - i0);
    if (threadIdx.x < kGroup) corr[threadIdx.x] = kap[threadIdx.x] - (kap[0] + threadIdx.x * dk);
    for (int e = threadIdx.x; e < ne; e += kTgt) {
        const double2 d = dz[vo0 + i0 + e];
        const double sp = sqrt(d.x * d.x + d.y * d.y) * wq;
        zs[e] = z[vo0 + i0 + e];
        for (int j = 0; j < cnt; ++j) {
            const double2 q = psi[t.vec_off[s0 + j] + i0 + e];
            const double f = sp * isqk[j];
            ps[j][e] = make_double2(q.x * f, q.y * f);
        }
    }
    __syncthreads();
    const int it = blockIdx.x * kTileF64 + threadIdx.x % kTileF64;
    double2 acc[kGroup];
#pragma unroll
    for (int j = 0; j < kGroup; ++j) acc[j] = make_double2(0.0, 0.0);
    if (it < n_x) {
        const double px = x[2 * it], py = x[2 * it + 1];
        for (int e = threadIdx.x / kTileF64; e < ne; e += kSlicesF64) {
            const double d1 = px - zs[e].x, d2 = py - zs[e].y;
            const double r = sqrt(d1 * d1 + d2 * d2);
            const double ir = 1.0 / r;
            const double ar = sqrt(kTwoOverPi * ir) * kSqrtHalf;
            double sn, cs, ss, sc;
            sincos(kap[0] * r, &sn, &cs);
            sincos(dk * r, &ss, &sc);
            double c0 = (cs + sn) * ar, s0v = (sn - cs) * ar;   // sqrt(2/(pi r)) e^{i(x0 - pi/4)}
            const float rf = (float)r;
            const double lnr = kapf[0] * rf < 8.f ? log(r) : 0.0;   // shared by the group
#pragma unroll
            for (int j = 0; j < kGroup; ++j) {
                if (j < cnt) {
                    const float xf = kapf[j] * rf;
                    double J0, Y0;   // times sqrt(kappa_j)
                    if (xf >= 8.f) {
                        const double dl = corr[j] * r;
                        const double c = fma(-dl, s0v, c0), sv = fma(dl, c0, s0v);
                        double P0, Q0, P1, Q1;
                        pq_horner<false>(pqt, xf, ir * ikap8[j], P0, Q0, P1, Q1);
                        J0 = fma(P0, c, -Q0 * sv);
                        Y0 = fma(P0, sv, Q0 * c);
                    } else {
                        bessel_small0_ln(kAS, kap[j] * r, lnk2[j] + lnr, J0, Y0);
                        J0 *= sqk[j];
                        Y0 *= sqk[j];
                    }
                    const double2 q = ps[j][e];
                    acc[j].x = fma(-Y0, q.x, fma(-J0, q.y, acc[j].x));
                    acc[j].y = fma(-Y0, q.y, fma(J0, q.x, acc[j].y));
                    const double cn = fma(c0, sc, -s0v * ss);
                    s0v = fma(s0v, sc, c0 * ss);
                    c0 = cn;
                }
            }
        }
    }
#pragma unroll
    for (int j = 0; j < kGroup; ++j) sums[j][threadIdx.x] = acc[j];
    __syncthreads();
    for (int o = threadIdx.x; o < cnt * kTileF64; o += kTgt) {
        const int j = o / kTileF64, k = o % kTileF64, ix = blockIdx.x * kTileF64 + k;
        if (ix >= n_x) continue;
        double2 v = sums[j][k];
#pragma unroll
        for (int sl = 1; sl < kSlicesF64; ++sl) {
            const double2 u = sums[j][sl * kTileF64 + k];
            v.x += u.x;
            v.y += u.y;
        }
        part[((long long)w * kGroup + j) * n_x + ix] = v;
    }
}

// Mixed-precision variant of field_partial_kernel: the same sums with the
// distances, H0 (Hankel form for kappa r >= 8, the small-argument series with
// ln r formed once per target-node pair below it), the phases and the
// accumulation in double-float arithmetic (the phases e^{i kappa_0 r} and
// e^{i dkappa r} reduced in binary32 pieces, FP64 only for kappa_0 r >= 6000).
// The amplitude sqrt(2 / (pi r)) rides on the phase of each target-node pair
// and 1 / sqrt(kappa_j) on the staged densities, so that the Hankel form
// returns sqrt(kappa_j) H0 and needs no amplitude product per frequency.
// Bound by FP32 issue.  The frequency loop works on pairs packed in one
// instruction: (cos, sin) of the phase, (P0, Q0), (J0, Y0) and (re, im) of the
// sums.  The correction corr_j r of the phase is applied as its increment from
// the frequency before, so that one exchange of (cos, sin) serves the Hankel
// form and the step.
// A CTA takes kTileDf targets, thread (target tid % 32, slice tid / 32) every
// fourth node of the chunk, and the slices' sums are added in slice order: the
// grid has four times the CTAs of one target per thread, each a quarter as
// long, which is what a few hundred targets (one problem of a batch) need.
// Measured (GB300): 1024 targets x 511 frequencies, N up to 1920: 7.6 -> 6.7 ms;
// x 255, N up to 480: 1.21 -> 0.93 ms (FMA pipe 69 %); 256 targets of each of 16 obstacles (127
// frequencies, N 64..832): 8.3 -> 3.5 ms.
constexpr int kTileDf = 32, kSlicesDf = kTgt / kTileDf;

template <int kG>   // largest subgroup size of the launch (<= kGroup)
__global__ void __launch_bounds__(kTgt, 6) field_partial_df_kernel(
    SolveTables t, Subgroups grp, const int2 *__restrict__ items, int item_begin, int chunk,
    const double2 *__restrict__ z, const double2 *__restrict__ dz,
    const double2 *__restrict__ psi, const double *__restrict__ x, int n_x,
    const float4 *__restrict__ zf, double2 *__restrict__ part) {
    const int w = blockIdx.y;
    const int2 item = items[item_begin + w];
    const int g = item.x, i0 = item.y;
    const int2 sgv = grp.sg[g];
    const int s0 = sgv.x, cnt = sgv.y;
    const int N = t.N[s0];
    const int vo0 = t.vec_off[s0];
    const double wq = 2.0 * kPi / (double)N * 0.25;   // (pi/n) / 4
    const double dk = grp.dkappa[g];
    const dfv dkd = df_from(dk);
    const float dkf = (float)dk;
    __shared__ double kap0;
    __shared__ float kapf[kGroup], dcorr[kGroup];
    __shared__ dfv ikap8[kGroup], sqk[kGroup], kapd[kGroup], lnk2[kGroup];
    __shared__ double isqd[kGroup];
    __shared__ float k3s[3];   // kappa_0 as three binary32 pieces
    __shared__ float4 zs[kChunk];             // node coordinates, double-float
    // q = (pi/n)|z'|/4 psi_j / sqrt(kappa_j) as (-re, -im) and (-im, re): (hi, hi, lo, lo)
    __shared__ float4 ps[kG][kChunk][2];
    // each thread's sums (re, im) per frequency, hi and lo, in its own column:
    // the frequency loop stays rolled (a small instruction footprint)
    __shared__ float2 accs[kG][2][kTgt];
    __shared__ GPair<1> gt;
    __shared__ float4 as[kAS_NI * kASPair];
    g_stage_pairs<1>(gt, {0}, {1});
    for (int e = threadIdx.x; e < kAS_NI * kASPair; e += kTgt) as[e] = reinterpret_cast<const float4 *>(kASJY0)[e];
    if (threadIdx.x == 0) {
        const double k0 = t.kappa[s0];
        const float a = (float)k0, b = (float)(k0 - (double)a);
        kap0 = k0;
        k3s[0] = a;
        k3s[1] = b;
        k3s[2] = (float)(k0 - (double)a - (double)b);
    }
    if (threadIdx.x < kGroup) {
        const int j = threadIdx.x;
        const double k0 = t.kappa[s0];
        const double k = (j < cnt) ? t.kappa[s0 + j] : 1.0;
        kapf[j] = (float)k;
        ikap8[j] = df_from(8.0 / k);
        sqk[j] = df_from(sqrt(k));
        isqd[j] = 1.0 / sqrt(k);
        kapd[j] = df_from(k);
        lnk2[j] = df_from(log(0.5 * k));   // ln(kappa/2): ln(x/2) = ln(kappa/2) + ln r
        // kappa_j - kappa_{j-1} - dkappa: the phase's correction beyond the step
        dcorr[j] = (j > 0 && j < cnt) ? (float)((k - (k0 + j * dk)) - (t.kappa[s0 + j - 1] - (k0 + (j - 1) * dk))) : 0.f;
    }
    __syncthreads();
    const int ne = min(chunk, N - i0);
    for (int e = threadIdx.x; e < ne; e += kTgt) {
        const double2 d = dz[vo0 + i0 + e];
        const double sp = sqrt(d.x * d.x + d.y * d.y) * wq;
        zs[e] = zf[vo0 + i0 + e];
        for (int j = 0; j < cnt; ++j) {
            const double2 q = psi[t.vec_off[s0 + j] + i0 + e];
            const double spj = sp * isqd[j];
            const dfv re = df_from(q.x * spj), im = df_from(q.y * spj);
            ps[j][e][0] = make_float4(-re.hi, -im.hi, -re.lo, -im.lo);
            ps[j][e][1] = make_float4(-im.hi, re.hi, -im.lo, re.lo);
        }
    }
    for (int j = 0; j < cnt; ++j) accs[j][0][threadIdx.x] = accs[j][1][threadIdx.x] = p2(0.f, 0.f);
    __syncthreads();
    const int it = blockIdx.x * kTileDf + threadIdx.x % kTileDf;
    if (it < n_x) {
        const dfv npx = df_neg(df_from(x[2 * it])), npy = df_neg(df_from(x[2 * it + 1]));
        const dfv two_over_pi = df_make(0.6366197466850281f, 2.5682552973194106e-08f);   // 2/pi
        for (int e = threadIdx.x / kTileDf; e < ne; e += kSlicesDf) {
            const float4 z4 = zs[e];
            const dfv d1 = df_add(df_make(z4.x, z4.y), npx), d2 = df_add(df_make(z4.z, z4.w), npy);
            const dfv rd = df_sqrt(df_add(df_mul(d1, d1), df_mul(d2, d2)));
            const dfv ir = df_rcp(rd);
            const dfv amp0 = df_sqrt(df_mul(ir, two_over_pi));   // sqrt(2 / (pi r))
            dfv c, sv, sc, ss;
            if (kapf[0] * rd.hi < kExpiKrMax) df_expi_kr(k3s[0], k3s[1], k3s[2], rd, c, sv);
            else df_expi_cold(kap0 * df_to(rd) - 0.78539816339744830962, c, sv);   // e^{i (kappa_0 r - pi/4)}
            if (dkf * rd.hi < 3.1f) df_sincos_mid(df_mul(dkd, rd), ss, sc);   // e^{i dkappa r}, no FP64 reduction
            else df_expi_cold(dk * df_to(rd), sc, ss);
            df2 cs = df2_mul(df2_make(c, sv), df2_bcast(amp0));
            const df2 stc = df2_bcast(sc), sts = df2_make(df_neg(ss), ss);
            const dfv lnr = kapf[0] * rd.hi < 8.0f ? df_log(rd) : df_make(0.f, 0.f);   // shared by the group
            const bool renorm = ((e / kSlicesDf) & 15) == 15;
#pragma unroll 1
            for (int j = 0; j < cnt; ++j) {
                const float xf = kapf[j] * rd.hi;
                const float dl = dcorr[j] * rd.hi;
                cs = df2_add_f(cs, p2(-dl * cs.h.y, dl * cs.h.x));
                const df2 sw = df2_swap(cs);
                df2 JY;   // sqrt(kappa_j) (J0, Y0)
                if (xf >= 8.0f) {
                    JY = df2_hankel0(gt, xf, df_mul(ir, ikap8[j]), cs, sw);
                } else {
                    JY = df2_mul(df2_bessel_small0(as, df_mul(kapd[j], rd), df_add(lnr, lnk2[j])), df2_bcast(sqk[j]));
                }
                // sums += Y0 (-qr, -qi) + J0 (-qi, qr)
                const float4 qy = ps[j][e][0], qj = ps[j][e][1];
                float2 h = accs[j][0][threadIdx.x], l = accs[j][1][threadIdx.x];
                df2_acc(h, l, df2_bcast(df2_y(JY)), {p2(qy.x, qy.y), p2(qy.z, qy.w)});
                df2_acc(h, l, df2_bcast(df2_x(JY)), {p2(qj.x, qj.y), p2(qj.z, qj.w)});
                if (renorm) {   // every 16 nodes of the thread
                    const df2 v = df2_quick(h, l);
                    h = v.h;
                    l = v.l;
                }
                accs[j][0][threadIdx.x] = h;
                accs[j][1][threadIdx.x] = l;
                cs = df2_dot2(cs, stc, sw, sts);   // c' = c cos - s sin, s' = s cos + c sin
            }
        }
    }
    __syncthreads();
    for (int o = threadIdx.x; o < cnt * kTileDf; o += kTgt) {
        const int j = o / kTileDf, k = o % kTileDf, ix = blockIdx.x * kTileDf + k;
        if (ix >= n_x) continue;
        double2 v = make_double2(0.0, 0.0);
#pragma unroll
        for (int sl = 0; sl < kSlicesDf; ++sl) {
            const float2 h = accs[j][0][sl * kTileDf + k], l = accs[j][1][sl * kTileDf + k];
            v.x += (double)h.x + (double)l.x;
            v.y += (double)h.y + (double)l.y;
        }
        part[((long long)w * kGroup + j) * n_x + ix] = v;
    }
}

// V[solve_j[s0 + j]][x] = sum over the subgroup's items, in item order.
__global__ void field_reduce_kernel(Subgroups grp, int g_begin, const int *__restrict__ item_first,
                                    int item_begin, const int *__restrict__ solve_j,
                                    const double2 *__restrict__ part, int n_x,
                                    double2 *__restrict__ V) {
    const int g = g_begin + blockIdx.y;
    const int it = blockIdx.x * blockDim.x + threadIdx.x;
    if (it >= n_x) return;
    const int2 sgv = grp.sg[g];
    const int w0 = item_first[g] - item_begin, w1 = item_first[g + 1] - item_begin;
    for (int j = 0; j < sgv.y; ++j) {
        double2 acc = make_double2(0.0, 0.0);
        for (int w = w0; w < w1; ++w) {
            const double2 v = part[((long long)w * kGroup + j) * n_x + it];
            acc.x += v.x;
            acc.y += v.y;
        }
        V[(long long)solve_j[sgv.x + j] * n_x + it] = acc;
    }
}

__global__ void field_zero_freq_kernel(int n_x, double2 *__restrict__ V) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n_x) V[i] = make_double2(1.0, 0.0);
}

__global__ void bessel_eval_kernel(const double *__restrict__ x, int n, double *__restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double J0, Y0, J1, Y1;
    bessel_j0y0j1y1(x[i], J0, Y0, J1, Y1);
    double a, b;
    bessel_j0y0(x[i], a, b);
    out[6 * i + 0] = J0;
    out[6 * i + 1] = Y0;
    out[6 * i + 2] = J1;
    out[6 * i + 3] = Y1;
    out[6 * i + 4] = a;
    out[6 * i + 5] = b;
}

// J0, Y0, J1, Y1 through the double-float routines of the mixed-precision
// kernels (Hankel form for x >= 8, small-argument series with a double-float
// logarithm below), for testing them.
__global__ void bessel_eval_df_kernel(const double *__restrict__ x, int n, double *__restrict__ out) {
    __shared__ GPair<2> gt;
    g_stage_pairs<2>(gt, {0, 1}, {2, 3});
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double xv = x[i];
    const dfv r8 = df_from(8.0 / xv);
    df2 J, N;
    if (xv >= 8.0) {
        dfv c, s;
        df_expi(xv - 0.78539816339744830962, c, s);
        const df2 cs = df2_mul(df2_make(c, s), df2_bcast(df_from(sqrt(kTwoOverPi / xv))));   // amplitude carried by the phase
        df2_hankel01(gt, (float)xv, r8, cs, df2_swap(cs), J, N);
    } else {
        const dfv xd = df_from(xv);
        const dfv lnh = df_add(df_log(xd), df_make(kLogConstDF[4], kLogConstDF[5]));   // ln(x/2)
        df2_bessel_small01(reinterpret_cast<const float4 *>(kASJY01), xd, r8, lnh, J, N);
    }
    out[4 * i + 0] = df_to(df2_x(J));
    out[4 * i + 1] = -df_to(df2_x(N));
    out[4 * i + 2] = df_to(df2_y(J));
    out[4 * i + 3] = -df_to(df2_y(N));
}

}  // namespace

void launch_bessel_eval(const double *x, int n, double *out, cudaStream_t st) {
    if (n > 0) bessel_eval_kernel<<<(n + 127) / 128, 128, 0, st>>>(x, n, out);
}

void launch_bessel_eval_df(const double *x, int n, double *out, cudaStream_t st) {
    if (n > 0) bessel_eval_df_kernel<<<(n + 127) / 128, 128, 0, st>>>(x, n, out);
}

void launch_target_field(const SolveTables &t, const Subgroups &g, int g_begin, int n_groups,
                         const int2 *items, int item_begin, int n_items, int chunk,
                         int group_max, const int *item_first, const int *solve_j,
                         const double2 *z, const double2 *dz, const double2 *psi, const double *x,
                         int n_x, const float4 *zf, double2 *part, double2 *V, bool double_float,
                         cudaStream_t st) {
    if (n_x <= 0) return;
    field_zero_freq_kernel<<<(n_x + 255) / 256, 256, 0, st>>>(n_x, V);
    if (n_groups <= 0 || n_items <= 0) return;
    const dim3 grid((n_x + kTileDf - 1) / kTileDf, n_items);
    if (double_float && group_max <= 4)
        field_partial_df_kernel<4><<<grid, kTgt, 0, st>>>(t, g, items, item_begin, chunk, z, dz, psi, x,
                                                          n_x, zf, part);
    else if (double_float)
        field_partial_df_kernel<kGroup><<<grid, kTgt, 0, st>>>(t, g, items, item_begin, chunk, z, dz, psi,
                                                               x, n_x, zf, part);
    else
        field_partial_kernel<<<dim3((n_x + kTileF64 - 1) / kTileF64, n_items), kTgt, 0, st>>>(
            t, g, items, item_begin, chunk, z, dz, psi, x, n_x, part);
    dim3 g2((n_x + 127) / 128, n_groups);
    field_reduce_kernel<<<g2, 128, 0, st>>>(g, g_begin, item_first, item_begin, solve_j, part, n_x, V);
}

}  // namespace fh
