// Step a2: Nystrom assembly of the direct CFIE (Sec. 2.3, eq. CFIE_direct)
//
//   (1/2) psi + K* psi - i eta S psi = dB/dn - i eta B,  B = e^{i kappa p.r},
//
// with the logarithmic splitting of the S and K* kernels and Kress's weights
// R_d for ln(4 sin^2((t - tau)/2)) (the discretisation the paper cites as
// Colton & Kress Sec. 3.5).  With r = |z_l - z_i|, s = |z'|,
// N_il = z2'_i (z1_l - z1_i) - z1'_i (z2_l - z2_i):
//   M  = (i/4) H0(kappa r) s_l          M1 = -J0(kappa r) s_l / (4 pi)
//   L  = (i kappa/4) H1(kappa r)/r N_il s_l/s_i
//   L1 = -(kappa/4pi) J1(kappa r)/r N_il s_l/s_i
//   M2 = M - M1 ln(4 sin^2),  L2 = L - L1 ln(4 sin^2)
//   A  = I/2 + R o (L1 - i eta M1) + (pi/n)(L2 - i eta M2)
// Diagonal limits: M1 = -s/4pi, M2 = [i/4 - C/2pi - ln(kappa s/2)/2pi] s,
// L1 = 0, L2 = (z1'' z2' - z2'' z1') / (4 pi s^2).
//
// One CTA assembles one 32 x 32 tile of the upper triangle, and its mirror
// image, for up to kGroup frequencies; tiles of all frequencies (of all
// problems of a batch) form one flat launch (prefix offsets tile_off).  Each
// warp writes 32 consecutive rows of a column (512 B) and the transposed
// entries, 16 B per row, which meet in L2.
#include "bessel.cuh"
#include "dfloat.cuh"
#include "fh_internal.h"

namespace fh {
namespace {

constexpr int kTile = 32;
constexpr int kNearBand = 2;   // off-diagonals whose special functions stay FP64 (mixed paths)

__device__ __forceinline__ int find_solve(const long long *__restrict__ off, int S, long long b) {
    int lo = 0, hi = S;  // off[lo] <= b < off[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= b) lo = mid; else hi = mid;
    }
    return lo;
}

// Upper-triangle tile of flat index lt: lt = tc (tc + 1) / 2 + tr, 0 <= tr <= tc.
__device__ __forceinline__ void triangle_tile(long long lt, int &tr, int &tc) {
    int c = (int)((sqrtf(8.f * (float)lt + 1.f) - 1.f) * 0.5f);
    while (c > 0 && (long long)c * (c + 1) / 2 > lt) --c;
    while ((long long)(c + 1) * (c + 2) / 2 <= lt) ++c;
    tc = c;
    tr = (int)(lt - (long long)c * (c + 1) / 2);
}

// FP64 assembly.  Per node pair and frequency, with
//   g4 = N_il s_l / (4 s_i r),  s4 = s_l / 4,  W = (pi/n) ln(4 sin^2) - R,
//   A1 = g4 W/pi, B1 = g4 pi/n, C1 = s4 pi/n, D1 = s4 W/pi,
//   Re A = kappa (A1 J1 - B1 Y1) + eta C1 J0,  Im A = kappa B1 J1 + eta (C1 Y0 - D1 J0)
// (the combination of M, M1, M2, L, L1, L2 above).  r, the Bessel values and W
// (even in i - l) are those of A(l, i) too, so a CTA takes a 32 x 32 tile of
// the upper triangle for up to kGroup frequencies of one N and writes both
// entries of every pair, the second one with its own geometry factors (N_li,
// s_i and s_l exchanged).  Once per pair: the geometry factors, the phase
// e^{i(kappa_0 r - pi/4)} with the amplitude sqrt(2 / (pi r)), the step e^{i
// dkappa r}, and ln r where the small-argument series will need it.
// Bound by the FP64 pipe (2 FMAs per clock and SM): about 75 FP64 instructions
// per entry, the small-argument series of the near-diagonal warps included,
// against 168 for one thread per entry with M1, M2, L1, L2 formed separately.
// Measured (GB300): 255 systems of N 64..480: 5.75 -> 2.32 ms (FP64 pipe active 90 %
// of the cycles; 3.56 ms with Clenshaw sums below x = 8 and FP64 interval
// comparisons); 63 systems of N = 256: 1.77 -> 0.65 ms.
__global__ void __launch_bounds__(256, 2) assemble_group_kernel(
    SolveTables t, Subgroups grp, int n_groups, const double2 *__restrict__ z,
    const double2 *__restrict__ dz, const double2 *__restrict__ ddz,
    const double *__restrict__ kress, const double *__restrict__ logsin,
    double2 *__restrict__ A, long long out_shift, long long tile_base) {
    const long long b = tile_base + blockIdx.x;
    const int g = find_solve(grp.tile_off, n_groups, b);
    const int2 sgv = grp.sg[g];
    const int s0 = sgv.x, cnt = sgv.y;
    const int N = t.N[s0];
    int tr, tc;
    triangle_tile(b - grp.tile_off[g], tr, tc);
    __shared__ double kap[kGroup], eta[kGroup], ikap8[kGroup], sqk[kGroup], eqk[kGroup], lnk2[kGroup], corr[kGroup];
    __shared__ float kapf[kGroup];
    __shared__ long long moff[kGroup];
    __shared__ PQShared pqt;
    pq_stage(pqt);
    const double dk = grp.dkappa[g];
    if (threadIdx.x < kGroup) {
        const int j = threadIdx.x;
        const double k = (j < cnt) ? t.kappa[s0 + j] : 1.0;
        const double e = (j < cnt) ? t.eta[s0 + j] : 0.0;
        kap[j] = k;
        kapf[j] = (float)k;
        eta[j] = e;
        ikap8[j] = 8.0 / k;
        sqk[j] = sqrt(k);
        eqk[j] = e / sqrt(k);
        lnk2[j] = log(0.5 * k);
        moff[j] = ((j < cnt) ? t.mat_off[s0 + j] : 0) + out_shift;
    }
    __syncthreads();
    if (threadIdx.x < kGroup) corr[threadIdx.x] = kap[threadIdx.x] - (kap[0] + threadIdx.x * dk);
    __syncthreads();
    const int i = tr * kTile + (threadIdx.x & 31);
    if (i >= N) return;
    const int vo = t.vec_off[s0];
    const int to = t.tab_off[t.tab[s0]];
    const double pin = 2.0 * kPi / (double)N;   // pi / n
    const double2 zi = z[vo + i], dzi = dz[vo + i];
    const double si = sqrt(dzi.x * dzi.x + dzi.y * dzi.y);
    const double inv4pi = 1.0 / (4.0 * kPi);
    const double isi = 1.0 / si, si4 = 0.25 * si, C2 = si4 * pin;

    for (int q = threadIdx.x >> 5; q < kTile; q += 8) {
        const int l = tc * kTile + q;
        if (l >= N) break;
        if (tr == tc && l < i) continue;   // each pair once on a diagonal tile
        int d = i - l;
        if (d < 0) d += N;
        const double Rw = kress[to + d];
        const long long e_il = (long long)l * N + i, e_li = (long long)i * N + l;
        if (l == i) {
            const double2 dd = ddz[vo + i];
            const double M1 = -si * inv4pi;
            const double L2r = (dd.x * dzi.y - dd.y * dzi.x) * inv4pi / (si * si);
            for (int j = 0; j < cnt; ++j) {
                const double M2r = (-kEulerGamma / (2.0 * kPi) - log(kap[j] * si * 0.5) / (2.0 * kPi)) * si;
                const double M2i = 0.25 * si;
                const double ar = 0.5 + pin * (L2r + eta[j] * M2i);
                const double ai = Rw * (-eta[j] * M1) + pin * (0.0 - eta[j] * M2r);
                A[moff[j] + e_il] = make_double2(ar, ai);
            }
            continue;
        }
        const double2 zl = z[vo + l], dzl = dz[vo + l];
        const double d1 = zl.x - zi.x, d2 = zl.y - zi.y;
        const double r = sqrt(d1 * d1 + d2 * d2);
        const double ir = 1.0 / r;
        const double sl = sqrt(dzl.x * dzl.x + dzl.y * dzl.y);
        const double sl4 = 0.25 * sl;
        const double Wp = fma(pin, logsin[to + d], -Rw) * (1.0 / kPi);   // W / pi
        const double g4 = (dzi.y * d1 - dzi.x * d2) * sl4 * isi * ir;     // N_il s_l / (4 s_i r)
        const double h4 = (dzl.x * d2 - dzl.y * d1) * si4 / sl * ir;      // N_li s_i / (4 s_l r)
        const double A1 = g4 * Wp, B1 = g4 * pin, C1 = sl4 * pin, D1 = sl4 * Wp;
        const double A2 = h4 * Wp, B2 = h4 * pin, D2 = si4 * Wp;
        const double amp = sqrt(kTwoOverPi * ir);
        double sn, cs, ss, sc;
        sincos(kap[0] * r, &sn, &cs);
        sincos(dk * r, &ss, &sc);
        const double ah = amp * kSqrtHalf;
        double c0 = (cs + sn) * ah, s0v = (sn - cs) * ah;   // amp e^{i(x0 - pi/4)}
        const float rf = (float)r;
        const double lnr = kapf[0] * rf < 8.f ? log(r) : 0.0;   // shared by the group
#pragma unroll 1
        for (int j = 0; j < cnt; ++j) {
            const float xf = kapf[j] * rf;
            const double r8 = ir * ikap8[j];
            double J0, Y0, J1, Y1;   // times sqrt(kappa_j)
            if (xf >= 8.f) {
                const double dl = corr[j] * r;
                const double c = fma(-dl, s0v, c0), sv = fma(dl, c0, s0v);
                double P0, Q0, P1, Q1;
                pq_horner<true>(pqt, xf, r8, P0, Q0, P1, Q1);
                J0 = fma(P0, c, -Q0 * sv);
                Y0 = fma(P0, sv, Q0 * c);
                J1 = fma(P1, sv, Q1 * c);
                Y1 = fma(Q1, sv, -P1 * c);
            } else {
                bessel_small_ln(kAS, kap[j] * r, r8, lnk2[j] + lnr, J0, Y0, J1, Y1);
                const double f = sqk[j];
                J0 *= f;
                Y0 *= f;
                J1 *= f;
                Y1 *= f;
            }
            J0 *= eqk[j];
            Y0 *= eqk[j];
            J1 *= sqk[j];
            Y1 *= sqk[j];
            double2 *Aj = A + moff[j];
            Aj[e_il] = make_double2(fma(A1, J1, fma(C1, J0, -B1 * Y1)), fma(B1, J1, fma(C1, Y0, -D1 * J0)));
            Aj[e_li] = make_double2(fma(A2, J1, fma(C2, J0, -B2 * Y1)), fma(B2, J1, fma(C2, Y0, -D2 * J0)));
            const double cn = fma(c0, sc, -s0v * ss);
            s0v = fma(s0v, sc, c0 * ss);
            c0 = cn;
        }
    }
}

// Mixed-precision variant of assemble_group_kernel.  With
//   k4 = kappa N_il s_l / (4 s_i r),  e4 = eta s_l / 4,
//   W  = (pi/n) ln(4 sin^2((t_i - t_l)/2)) - R_{i-l},
// the off-diagonal entry is
//   Re A = k4 (W/pi J1 - (pi/n) Y1) + (pi/n) e4 J0,
//   Im A = (pi/n) k4 J1 + e4 ((pi/n) Y0 - W/pi J0),
// the same combination of M, M1, M2, L, L1, L2 as the FP64 kernel.  For
// entries off the band |i - l| <= kNearBand, the Bessel values (Hankel form
// for kappa r >= 8, the small-argument series with ln r formed once per node
// pair below it), the phases and this combination run in double-float
// arithmetic; the diagonal and the band (where ln r and the Kress log table
// nearly cancel), the Kress weights and the log table stay FP64.  Entries are
// stored as double-float pairs (re hi, re lo, im hi, im lo): the FP32 LU takes
// the hi parts and the refinement residual uses both.  Per node pair the
// amplitude sqrt(2 / (pi r)) rides on the phase and the geometry factors are
// combined once,
//   A1 = g4 W/pi, B1 = g4 pi/n, C1 = s4 pi/n, D1 = s4 W/pi
//   (g4 = N_il s_l / (4 s_i r), s4 = s_l / 4),
// so that with J' = sqrt(kappa_j) J (what the Hankel form returns)
//   Re A = sqrt(kappa) (A1 J1' - B1 Y1') + (eta / sqrt(kappa)) C1 J0',
//   Im A = sqrt(kappa) B1 J1' + (eta / sqrt(kappa)) (C1 Y0' - D1 J0').
// Bound by FP32 issue: the frequency loop works on pairs packed in one
// instruction, (cos, sin) of the phase, (P0, P1) and (Q0, Q1), (J0, J1) and (Y0,
// Y1), and the two entries (i, l), (l, i).  With 8 points per wavelength about
// twenty entries of every row take the small-argument series (x < 8), whose
// warps cost as much as the others only with short series.
// Measured (GB300, band kernel and right sides included): 255 systems of N
// 64..480: 0.84 -> 0.51 ms; 511 systems of N 64..1920: 11.7 -> 10.1 ms; 16 x 127
// systems of N 64..832: 6.4 -> 4.1 ms.
// r, the Bessel values, the phases and the Kress log weight (even in i - l)
// are the same for A(i, l) and A(l, i): a CTA takes a tile (tr, tc) of the
// upper triangle (flat index tc (tc + 1) / 2 + tr within the subgroup) and
// writes both entries of every node pair (i < l on a diagonal tile), the
// second one with its own geometry factors (N_li, s_i, s_l swapped).  With
// A32 non-null the hi parts also go to the row-major FP32 copy that the
// tensor-core LU factors (A32(i, l) at i N + l, the same offsets as A).
__global__ void __launch_bounds__(256, 3) assemble_group_df_kernel(
    SolveTables t, Subgroups grp, int n_groups, const double2 *__restrict__ dz,
    const float4 *__restrict__ zf, const float4 *__restrict__ dzf, const float2 *__restrict__ sf,
    const float2 *__restrict__ wpf, float4 *__restrict__ A_out, float2 *__restrict__ A32, long long out_shift,
    long long tile_base) {
    const long long b = tile_base + blockIdx.x;
    const int g = find_solve(grp.tile_off, n_groups, b);
    const int2 sgv = grp.sg[g];
    const int s0 = sgv.x, cnt = sgv.y;
    const int N = t.N[s0];
    int tr, tc;
    triangle_tile(b - grp.tile_off[g], tr, tc);   // 0 <= tr <= tc < ceil(N / 32)
    __shared__ double kap0;
    __shared__ float kapf[kGroup], dcorr[kGroup];
    __shared__ dfv kapd[kGroup], ikap8[kGroup], sqk[kGroup], lnk2[kGroup];
    __shared__ df2 esq[kGroup];   // (eta / sqrt(kappa), sqrt(kappa))
    __shared__ long long moff[kGroup];
    __shared__ float k3s[3];   // kappa_0 as three binary32 pieces
    __shared__ GPair<2> gt;
    __shared__ float4 as[kAS_NI * 2 * kASPair];
    g_stage_pairs<2>(gt, {0, 1}, {2, 3});
    for (int e = threadIdx.x; e < kAS_NI * 2 * kASPair; e += blockDim.x) as[e] = reinterpret_cast<const float4 *>(kASJY01)[e];
    const double dk = grp.dkappa[g];
    const dfv dkd = df_from(dk);
    const float dkf = (float)dk;
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
        const double k = (j < cnt) ? t.kappa[s0 + j] : 1.0;
        const double e = (j < cnt) ? t.eta[s0 + j] : 0.0;
        const double k0 = t.kappa[s0];
        kapf[j] = (float)k;
        kapd[j] = df_from(k);
        ikap8[j] = df_from(8.0 / k);
        sqk[j] = df_from(sqrt(k));
        esq[j] = df2_make(df_from(e / sqrt(k)), sqk[j]);
        lnk2[j] = df_from(log(0.5 * k));   // ln(kappa/2): ln(x/2) = ln(kappa/2) + ln r
        // kappa_j - kappa_{j-1} - dkappa: the phase's correction beyond the step
        dcorr[j] = (j > 0 && j < cnt) ? (float)((k - (k0 + j * dk)) - (t.kappa[s0 + j - 1] - (k0 + (j - 1) * dk))) : 0.f;
        moff[j] = ((j < cnt) ? t.mat_off[s0 + j] : 0) + out_shift;
    }
    __syncthreads();
    const int i = tr * kTile + (threadIdx.x & 31);
    if (i >= N) return;
    const int vo = t.vec_off[s0];
    const int to = t.tab_off[t.tab[s0]];
    const double pin = 2.0 * kPi / (double)N;   // pi / n
    const dfv pind = df_from(pin);
    const double2 dzi = dz[vo + i];
    const double si = sqrt(dzi.x * dzi.x + dzi.y * dzi.y);
    const dfv isi4 = df_from(0.25 / si);
    const dfv two_over_pi = df_make(0.6366197466850281f, 2.5682552973194106e-08f);
    const float4 zi4 = zf[vo + i], dzi4 = dzf[vo + i];
    const dfv nzix = df_make(-zi4.x, -zi4.y), nziy = df_make(-zi4.z, -zi4.w);
    const dfv dzix = df_make(dzi4.x, dzi4.y), dziy = df_make(dzi4.z, dzi4.w);
    const float2 si2 = sf[vo + i];
    const dfv si4 = df_mul_f(df_make(si2.x, si2.y), 0.25f);   // s_i / 4
    const dfv C2 = df_mul(si4, pind);

    for (int q = threadIdx.x >> 5; q < kTile; q += 8) {
        const int l = tc * kTile + q;
        if (l >= N) break;
        if (tr == tc && l <= i) continue;   // each pair once on a diagonal tile
        int d = i - l;
        if (d < 0) d += N;
        if (d <= kNearBand || d >= N - kNearBand) continue;   // assemble_band_kernel
        const long long e_il = (long long)l * N + i, e_li = (long long)i * N + l;
        // pair geometry in double-float from the double-float node tables
        const float4 zl4 = zf[vo + l], dzl4 = dzf[vo + l];
        const dfv d1 = df_add(df_make(zl4.x, zl4.y), nzix), d2 = df_add(df_make(zl4.z, zl4.w), nziy);
        const dfv rd = df_sqrt(df_add(df_mul(d1, d1), df_mul(d2, d2)));
        const dfv ir = df_rcp(rd);
        const dfv Nil = df_add(df_mul(dziy, d1), df_neg(df_mul(dzix, d2)));
        // N_li = z2'_l (z1_i - z1_l) - z1'_l (z2_i - z2_l)
        const dfv Nli = df_dot2(df_make(dzl4.x, dzl4.y), d2, df_make(-dzl4.z, -dzl4.w), d1);
        const float2 sl2 = sf[vo + l], wp2 = wpf[to + d], wq2 = wpf[to + N - d];
        const dfv sl = df_make(sl2.x, sl2.y), Wp = df_make(wp2.x, wp2.y);   // |z'_l|, W / pi at i - l
        const dfv Wq = df_make(wq2.x, wq2.y);                                // W / pi at l - i
        const dfv gg4 = df_mul(df_mul(Nil, sl), df_mul(ir, isi4));          // N_il s_l / (4 s_i r)
        const dfv gq4 = df_mul(df_mul(Nli, si4), df_mul(ir, df_rcp(sl)));   // N_li s_i / (4 s_l r)
        const dfv sl4 = df_mul_f(sl, 0.25f);
        // (entry (i, l), entry (l, i))
        const df2 A = df2_mul(df2_make(gg4, gq4), df2_make(Wp, Wq)), B = df2_mul(df2_make(gg4, gq4), df2_bcast(pind));
        const df2 C = df2_make(df_mul(sl4, pind), C2), D = df2_mul(df2_make(sl4, si4), df2_make(Wp, Wq));
        const dfv amp0 = df_sqrt(df_mul(ir, two_over_pi));
        dfv c, sv, sc, ss;
        if (kapf[0] * rd.hi < kExpiKrMax) df_expi_kr(k3s[0], k3s[1], k3s[2], rd, c, sv);
        else df_expi_cold(kap0 * df_to(rd) - 0.78539816339744830962, c, sv);   // e^{i (kappa_0 r - pi/4)}
        if (dkf * rd.hi < 3.1f) df_sincos_mid(df_mul(dkd, rd), ss, sc);   // e^{i dkappa r}, no FP64 reduction
        else df_expi_cold(dk * df_to(rd), sc, ss);
        df2 cs = df2_mul(df2_make(c, sv), df2_bcast(amp0));
        const df2 stc = df2_bcast(sc), sts = df2_make(df_neg(ss), ss);
        const dfv lnr = kapf[0] * rd.hi < 8.0f ? df_log(rd) : df_make(0.f, 0.f);   // shared by the group
#pragma unroll 1   // not unrolled: half the registers, twice the occupancy
        for (int j = 0; j < cnt; ++j) {
            const float xf = kapf[j] * rd.hi, dl = dcorr[j] * rd.hi;
            cs = df2_add_f(cs, p2(-dl * cs.h.y, dl * cs.h.x));
            const df2 sw = df2_swap(cs);
            const dfv r8 = df_mul(ir, ikap8[j]);
            df2 J, Y;   // sqrt(kappa_j) (J0, J1) and -sqrt(kappa_j) (Y0, Y1)
            if (xf >= 8.0f) {
                df2_hankel01(gt, xf, r8, cs, sw, J, Y);
            } else {
                df2_bessel_small01(as, df_mul(kapd[j], rd), r8, df_add(lnr, lnk2[j]), J, Y);
                const df2 q = df2_bcast(sqk[j]);
                J = df2_mul(J, q);
                Y = df2_mul(Y, q);
            }
            J = df2_mul(J, esq[j]);   // (eta J0, kappa J1), and the same of -Y
            Y = df2_mul(Y, esq[j]);
            const df2 J0 = df2_bcast(df2_x(J)), J1 = df2_bcast(df2_y(J)), Y0 = df2_bcast(df2_x(Y)), Y1 = df2_bcast(df2_y(Y));
            const df2 re = df2_dot3(A, J1, B, Y1, C, J0);
            const df2 im = df2_dot3(B, J1, C, {p2_neg(Y0.h), p2_neg(Y0.l)}, D, {p2_neg(J0.h), p2_neg(J0.l)});
            const long long mo = moff[j];
            A_out[mo + e_il] = make_float4(re.h.x, re.l.x, im.h.x, im.l.x);
            A_out[mo + e_li] = make_float4(re.h.y, re.l.y, im.h.y, im.l.y);
            if (A32) {
                A32[mo + e_li] = make_float2(re.h.x, im.h.x);
                A32[mo + e_il] = make_float2(re.h.y, im.h.y);
            }
            cs = df2_dot2(cs, stc, sw, sts);   // c' = c cos - s sin, s' = s cos + c sin
        }
    }
}

// The diagonal and the band 0 < |i - l| <= kNearBand (cyclically) of the
// matrices of solves list[0 .. gridDim.y - 1] for the mixed paths, in
// FP64 with the FP64 kernel's formulas: there r is of the order of the node
// spacing and ln r nearly cancels against the Kress log table.  One thread
// per diagonal entry and per node pair (i, i + o), whose Bessel values serve
// both entries, so that no warp of assemble_group_df_kernel runs FP64 Bessel
// series for a few lanes.  A32 (may be null): the hi parts, row-major.
// Bound by the FP64 pipe: 16 x 127 systems of N 64..832 1175 -> 518 us, 511 of
// N 64..1920 1056 -> 471 us (one thread per entry before).
__global__ void __launch_bounds__(256) assemble_band_kernel(
    SolveTables t, const int *__restrict__ list, const double2 *__restrict__ z, const double2 *__restrict__ dz,
    const double2 *__restrict__ ddz, const double *__restrict__ kress,
    const double *__restrict__ logsin, float4 *__restrict__ A, float2 *__restrict__ A32, long long out_shift) {
    const int s = list[blockIdx.y];
    const int N = t.N[s];
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= N * (kNearBand + 1)) return;
    const int o = e / N, i = e - o * N;   // o = 0: the diagonal (whole warps take one branch)
    int l = i + o;
    if (l >= N) l -= N;
    const int vo = t.vec_off[s], to = t.tab_off[t.tab[s]];
    const double kappa = t.kappa[s], et = t.eta[s];
    const double pin = 2.0 * kPi / (double)N;   // pi / n
    const double inv4pi = 1.0 / (4.0 * kPi);
    const double2 zi = z[vo + i], dzi = dz[vo + i];
    const double si = sqrt(dzi.x * dzi.x + dzi.y * dzi.y);
    auto put = [&](int row, int col, double ar, double ai) {
        const float4 v = df_pack(ar, ai);
        A[t.mat_off[s] + out_shift + (long long)col * N + row] = v;
        if (A32) A32[t.mat_off[s] + out_shift + (long long)row * N + col] = make_float2(v.x, v.z);
    };
    if (o == 0) {
        const double Rw = kress[to];
        const double2 dd = ddz[vo + i];
        const double M1 = -si * inv4pi;
        const double L2r = (dd.x * dzi.y - dd.y * dzi.x) * inv4pi / (si * si);
        const double M2r = (-kEulerGamma / (2.0 * kPi) - log(kappa * si * 0.5) / (2.0 * kPi)) * si;
        const double M2i = 0.25 * si;
        put(i, i, 0.5 + pin * (L2r + et * M2i), Rw * (-et * M1) + pin * (0.0 - et * M2r));
    } else {
        const double2 zl = z[vo + l], dzl = dz[vo + l];
        const double e1 = zl.x - zi.x, e2 = zl.y - zi.y;
        const double r = sqrt(e1 * e1 + e2 * e2);
        const double sl = sqrt(dzl.x * dzl.x + dzl.y * dzl.y);
        double J0, Y0, J1, Y1;
        bessel_j0y0j1y1(kappa * r, J0, Y0, J1, Y1);
        // the entry with weights Rw, ls at its index difference, source length s and normal factor gg
        auto entry = [&](int row, int col, double Rw, double ls, double sc, double gg) {
            const double Mr = -0.25 * Y0 * sc, Mi = 0.25 * J0 * sc;
            const double M1 = -J0 * sc * inv4pi;
            const double M2r = Mr - M1 * ls;
            const double Lr = -0.25 * kappa * Y1 * gg, Li = 0.25 * kappa * J1 * gg;
            const double L1 = -kappa * inv4pi * J1 * gg;
            const double L2r = Lr - L1 * ls;
            put(row, col, Rw * L1 + pin * (L2r + et * Mi), Rw * (-et * M1) + pin * (Li - et * M2r));
        };
        entry(i, l, kress[to + N - o], logsin[to + N - o], sl, (dzi.y * e1 - dzi.x * e2) * sl / (si * r));
        entry(l, i, kress[to + o], logsin[to + o], si, (dzl.x * e2 - dzl.y * e1) * si / (sl * r));
    }
}

// g_i = dB/dn - i eta B = i (kappa p.nu_i - eta) e^{i kappa p.z_i}
__global__ void rhs_kernel(SolveTables t, const double2 *__restrict__ z,
                           const double2 *__restrict__ dz, const int *__restrict__ prob,
                           const double2 *__restrict__ pdir, double2 *__restrict__ g) {
    const int s = blockIdx.y;
    const int N = t.N[s];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double2 pd = pdir[prob[s]];
    const double p0 = pd.x, p1 = pd.y;
    const int o = t.vec_off[s] + i;
    const double kappa = t.kappa[s], eta = t.eta[s];
    const double2 zi = z[o], d = dz[o];
    const double sp = sqrt(d.x * d.x + d.y * d.y);
    const double pn = (p0 * d.y - p1 * d.x) / sp;
    const double a = kappa * pn - eta;
    double sn, cs;
    sincos(kappa * (p0 * zi.x + p1 * zi.y), &sn, &cs);
    g[o] = make_double2(-a * sn, a * cs);
}

}  // namespace

void launch_assemble_groups(const SolveTables &t, const Subgroups &g, int n_groups,
                            long long tile_base, long long n_tiles, const int *band_list,
                            int band_count, int maxN,
                            const double2 *z, const double2 *dz,
                            const double2 *ddz, const double *kress, const double *logsin,
                            const float4 *zf, const float4 *dzf, const float2 *sf, const float2 *wpf,
                            double2 *A, float4 *Af, float2 *A32, long long out_shift, cudaStream_t st,
                            cudaStream_t band_st) {
    if (n_tiles <= 0 || n_groups <= 0) return;
    if (Af) {
        if (band_count > 0) {
            const dim3 grid((maxN * (kNearBand + 1) + 255) / 256, band_count);
            assemble_band_kernel<<<grid, 256, 0, band_st>>>(t, band_list, z, dz, ddz, kress, logsin, Af,
                                                            A32, out_shift);
        }
        assemble_group_df_kernel<<<(unsigned)n_tiles, 256, 0, st>>>(t, g, n_groups, dz, zf, dzf, sf,
                                                                    wpf, Af, A32, out_shift, tile_base);
    } else
        assemble_group_kernel<<<(unsigned)n_tiles, 256, 0, st>>>(t, g, n_groups, z, dz, ddz, kress,
                                                                 logsin, A, out_shift, tile_base);
}

void launch_rhs(const SolveTables &t, int S, int maxN, const double2 *z, const double2 *dz,
                const int *prob, const double2 *pdir, double2 *g, cudaStream_t st) {
    if (S <= 0) return;
    dim3 grid((maxN + 127) / 128, S);
    rhs_kernel<<<grid, 128, 0, st>>>(t, z, dz, prob, pdir, g);
}

}  // namespace fh
