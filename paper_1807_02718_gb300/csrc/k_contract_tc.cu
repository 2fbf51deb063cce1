// Step a7 on the tensor cores: u[x][t] = sum_{kk < 2J} A[x][kk] B[kk][t] with
// A = [Vr | Vi] and B = [Gr ; Gm] (Sec. 4.1 eq. approx in collapsed form),
// to FP64 accuracy through exact BF16 products (an error-free slicing of the
// operands, the "Ozaki scheme").  Every precision contracts here, and so does
// the split synthesis, unless the outputs are few (contract_small,
// contract_slices_fp64) or may not allocate: the FP64 pipe bounds the plain FP64
// kernel.  Measured,
// plain -> slices (five launches): 1024 x 4096 outputs, 2J = 512 3.62 -> 0.21 ms
// (MMAs at the measured BF16 rate 0.08 ms; the rest is slicing, 42 MB written
// and read back, and the epilogue, which cannot overlap the MMAs: TMEM holds
// one tile's levels), 2J = 1024 7.2 -> 0.37 ms, 333 x 1001, 2J = 402 334 -> 74 us.
//
// The balance below is taken over all targets and times of the call, and the call's
// size decides between this kernel and the FP64 ones: a sample's last bits depend on
// what else the call asks for (the fields and weights that enter do not).
//
// Scaling.  Term kk is first balanced by a power of two, A[x][kk] 2^d_kk times
// B[kk][t] 2^-d_kk, so that entries which meet small partners (the fields at
// frequencies outside the signal's band) do not set the scales: d_kk is half
// the difference of the exponents of the largest entries of B's row kk and of
// A's column kk, every target's row of A and time's column of B taken relative
// to its own largest entry.  Each row x is then scaled by 2^ea_x with ea_x the
// exponent of its largest entry and cut into kSlices = 8 slices of kSliceBits
// = 7 bits, A / 2^ea_x = sum_i a_i 2^-(7 (i + 1)) + O(2^-57), a_i integers with
// |a_0| <= 2^7 and |a_i| <= 2^6; likewise each column t of B.  These integers
// are exact in BF16 and their products in the FP32 accumulator; a level d =
// i + j sums at most kSlices pairs over a K segment of kSegK = 512 terms: TMEM
// holds one FP32 accumulator per level (kSlices x 64 = 512 columns, all of it).
// Levels stay below 2^24 and exact, except levels 6 and 7 when nearly all 512
// terms have one sign and both factors within 10 % of their maxima; they then
// lose units of 2^-56 of a sum of some 2^8 of the same measure.  After each K
// segment the epilogue joins the levels as integers, rounds once to FP64 and
// adds up the segments; at the end the sums take the
// factor 2^(ea_x + eb_t - 14).  The result differs from the exact product by
// the dropped slice pairs (i + j >= kSlices) and the remainders, about 2^-58 of
// max|row| max|column| per term after balancing.  Measured against quadruple
// precision (relative L2, 64 x 96 outputs, 2J = 80 .. 1024; plain FP64 sums in
// brackets): random operands 0.7-0.9e-16 (1.7-5.3e-16), Gaussian spectra with
// sigma of 5 % of the band 0.8-1.4e-16 (1.6-5.0e-16), those against fields that
// grow by six decades over the band 0.9-1.8e-16 (1.6-4.9e-16).
//
// Rows of A and columns of B with an infinity or NaN, and tiles whose waits
// gave up, are summed directly in FP64.
//
// Kernels: ozaki_scale_kernel (ea, eb; once for the balance and once
// after it), ozaki_balance_kernel (d_kk), ozaki_slice_kernel (slices in BF16, written directly in the MMA's
// shared-memory layout: per 128-row (A) or 64-row (B) tile and K chunk of 16,
// the eight slices' K-major core matrices in one contiguous block; A and B in
// one launch each), contract_tc_kernel (one CTA per 128 x 64 output tile, warp
// specialised over a four-stage pipeline: one thread bulk-copies each chunk's
// A and B blocks (48 KB), one thread issues the kind::f16 MMAs of every slice
// pair into its level's accumulator, eight epilogue warps combine the levels
// after each segment; mbarriers with bounded waits hand the stages over).
#include <cuda_bf16.h>

#include <climits>

#include "fh_internal.h"
#include "tc_gemm.cuh"

namespace fh {
namespace {

constexpr int kSlices = 8;
constexpr int kSliceBits = 7;
constexpr int kTM = 128;                 // output rows (x) per CTA = TMEM lanes
constexpr int kTN = 64;                  // output columns (t) per CTA
constexpr int kKC = 16;                  // K elements per staged chunk: one MMA K step (32 bytes)
constexpr int kKBytes = kKC * 2;
constexpr int kKPad = 64;                // K padding of the slice arrays
constexpr int kThr = 256, kScaleThr = 512;
constexpr int kASlice = kTM * kKBytes;   // bytes of one A slice chunk (4 KiB)
constexpr int kBSlice = kTN * kKBytes;   // bytes of one B slice chunk (2 KiB)
constexpr int kABlock = kSlices * kASlice, kBBlock = kSlices * kBSlice;   // 32 + 16 KiB per chunk
constexpr int kStage = kABlock + kBBlock;                                 // 48 KiB
constexpr int kStages = 4;
constexpr int kSmem = 1024 + kStages * kStage;
constexpr int kSegK = 512;                  // K per exact segment
constexpr int kCtaThreads = 384;            // producer (warp 0), MMA (warp 1), epilogue (warps 4 .. 11)
constexpr int kOutPitch = 33;               // output tile of an epilogue warp: 32 x 32, padded rows
constexpr long long kWaitLimit = 1LL << 22;
#ifdef FH_TEST_CONTRACT_GIVES_UP
constexpr bool kTestGivesUp = true;         // a test's build: every tile reports, after its last wait, that one ran out
#else
constexpr bool kTestGivesUp = false;
#endif
constexpr int kZeroExp = INT_MIN / 4;       // exponent of a zero; balance of a term that is zero throughout
constexpr int kNonFinite = INT_MAX;         // scale of a row or column with an infinity or NaN
static_assert(8 * 32 * kOutPitch * (int)sizeof(double) <= kStages * kStage, "output tiles fit the stages");

// Element (r, kk) of the operand whose rows are r: A rows are targets x (from
// V[kk][x] complex, real parts for kk < J, imaginary parts above), B rows are
// times t (from Gr[kk][t] for kk < J, Gm[kk - J][t] above).
struct Src {
    const double2 *V;        // A: V[j * rows + r]
    const double *G0, *G1;   // B: Gr, Gm [j * rows + r]
    int J, rows;
    __device__ __forceinline__ double at(int r, int kk) const {
        if (r >= rows || kk >= 2 * J) return 0.0;
        const int j = kk < J ? kk : kk - J;
        if (V) {
            const double2 v = V[(long long)j * rows + r];
            return kk < J ? v.x : v.y;
        }
        return (kk < J ? G0 : G1)[(long long)j * rows + r];
    }
};

// e with |v| < 2^e (the least such), kZeroExp for zero, kNonFinite for
// infinities and NaN; integer operations (the FP64 pipe is the slow one).
__device__ __forceinline__ int exp_of(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v) & ~(1ull << 63);
    const int be = (int)(b >> 52);
    if (be == 0x7FF) return kNonFinite;
    if (be) return be - 1022;
    return b ? 64 - __clzll((long long)b) - 1074 : kZeroExp;
}

// d[j], d[J + j]: the balance of the terms Vr Gr and Vi Gm of frequency j, with
// ea, eb the exponents of the rows' largest entries (rows with an infinity or
// NaN take no part).  One CTA per j reads its three rows.
__global__ void __launch_bounds__(kThr) ozaki_balance_kernel(Src a, Src b, const int *__restrict__ ea,
                                                             const int *__restrict__ eb, int *__restrict__ d) {
    __shared__ int part[kThr / 32][4];
    const int j = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int m[4] = {kZeroExp, kZeroExp, kZeroExp, kZeroExp};   // Vr, Vi, Gr, Gm
    auto take = [](int &mx, double v, int e0) {
        const int e = exp_of(v);
        if (e0 != kNonFinite && e != kZeroExp) mx = max(mx, e - e0);
    };
#pragma unroll 4
    for (int x = threadIdx.x; x < a.rows; x += kThr) {
        const double2 v = a.V[(long long)j * a.rows + x];
        const int e0 = ea[x];
        take(m[0], v.x, e0);
        take(m[1], v.y, e0);
    }
#pragma unroll 4
    for (int t = threadIdx.x; t < b.rows; t += kThr) {
        const int e0 = eb[t];
        take(m[2], b.G0[(long long)j * b.rows + t], e0);
        take(m[3], b.G1[(long long)j * b.rows + t], e0);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        m[i] = __reduce_max_sync(0xffffffffu, m[i]);
        if (lane == 0) part[warp][i] = m[i];
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        int ma = kZeroExp, mb = kZeroExp;
        for (int w = 0; w < kThr / 32; ++w) {
            ma = max(ma, part[w][threadIdx.x]);
            mb = max(mb, part[w][2 + threadIdx.x]);
        }
        d[threadIdx.x * a.J + j] = ma == kZeroExp || mb == kZeroExp ? kZeroExp : (mb - ma) >> 1;
    }
}

// e[r] with max_kk |src(r, kk)| 2^(+-d[kk]) < 2^e[r] (0 for a zero row,
// kNonFinite with an infinity or NaN); d may be null (no balance).  A CTA
// takes 32 rows: lane = row (consecutive rows are contiguous in both sources),
// the sixteen warps stride over the frequencies, two terms each (latency
// bound), then a shared-memory maximum.  The first actas CTAs take A.
__global__ void __launch_bounds__(kScaleThr) ozaki_scale_kernel(Src a, Src b, int actas, const int *__restrict__ d,
                                                                int *__restrict__ ea, int *__restrict__ eb) {
    __shared__ int part[kScaleThr / 32][32];
    const bool left = (int)blockIdx.x < actas;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, J = a.J;
    const int r = (left ? blockIdx.x : blockIdx.x - actas) * 32 + lane, rows = left ? a.rows : b.rows;
    int m = kZeroExp;
    auto take = [&](double v, int dk) {
        const int e = exp_of(v);
        if (e == kNonFinite) m = kNonFinite;
        else if (e != kZeroExp && dk != kZeroExp) m = max(m, left ? e + dk : e - dk);
    };
    if (r < rows) {
#pragma unroll 8
        for (int j = warp; j < J; j += kScaleThr / 32) {
            const long long o = (long long)j * rows + r;
            const double2 v = left ? __ldg(a.V + o) : make_double2(__ldg(b.G0 + o), __ldg(b.G1 + o));
            take(v.x, d ? __ldg(d + j) : 0);
            take(v.y, d ? __ldg(d + J + j) : 0);
        }
    }
    part[warp][lane] = m;
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int w = 1; w < kScaleThr / 32; ++w) m = max(m, part[w][lane]);
        (left ? ea : eb)[r] = m == kZeroExp ? 0 : m;
    }
}

// Slices of a 64-row x 32-column block, in BF16, written into the tiled
// layout the contraction copies in bulk: for tile rows tr (128 for A, 64 for
// B) and K chunks of 16, block (r / tr) * nkc + kk / 16 holds the eight slices
// one after the other, each tr rows of 32 bytes as K-major core matrices
// (8 rows x 16 bytes; the two 16-byte halves of K 128 bytes apart, 8-row
// groups 256 bytes apart).
// In integer arithmetic on the FP64 bit pattern: V = round(src 2^(+-d[kk] + 56
// - e[r])) (|V| <= 2^56) = sum_s a_s 2^(49 - 7 s) with balanced digits, each the
// nearest multiple of the remainder (|a_0| <= 128, |a_s| <= 64), so that the
// dropped slice products carry no common sign.  The first ablocks blocks of x take A.
__global__ void __launch_bounds__(kThr) ozaki_slice_kernel(Src sa, Src sb, int ablocks, const int *__restrict__ d,
                                                           const int *__restrict__ ea, const int *__restrict__ eb,
                                                           int kpad, __nv_bfloat16 *__restrict__ outa,
                                                           __nv_bfloat16 *__restrict__ outb) {
    __shared__ __nv_bfloat16 t[kSlices][32][64 + 8];   // [slice][kk][r], padded rows
    const bool left = (int)blockIdx.x < ablocks;
    const Src src = left ? sa : sb;
    const int *e = left ? ea : eb;
    const int r0 = (left ? blockIdx.x : blockIdx.x - ablocks) * 64, k0 = blockIdx.y * 32, tr = left ? kTM : kTN;
    for (int idx = threadIdx.x; idx < 64 * 32; idx += kThr) {
        const int rr = idx & 63, kk = idx >> 6;          // consecutive threads: consecutive rows
        const int r = r0 + rr, er = e[r], dk = k0 + kk < 2 * src.J ? d[k0 + kk] : kZeroExp;
        const unsigned long long bits = (unsigned long long)__double_as_longlong(src.at(r, k0 + kk));
        const int bexp = (int)((bits >> 52) & 0x7FF);
        const unsigned long long mant = (bits & ((1ull << 52) - 1)) | (bexp ? (1ull << 52) : 0ull);
        long long V = 0;
        if (er != kNonFinite && dk != kZeroExp && mant) {
            // |src| = mant 2^(bexp - 1075) (1 - 1075 for subnormals); mant 2^sh <= 2^56 by the choice of e[r]
            const int sh = (bexp ? bexp : 1) - 1075 + (left ? dk : -dk) + kSlices * kSliceBits - er;
            if (sh >= 0) V = (long long)(mant << sh);
            else if (sh > -64) V = (long long)((mant + (1ull << (-sh - 1))) >> -sh);   // round half up on |V|
        }
        if (bits >> 63) V = -V;
        // two halves of four digits each in 32-bit arithmetic
        const int vh = (int)((V + (1ll << 27)) >> 28);
        int v = vh;
#pragma unroll
        for (int s = 0; s < kSlices; ++s) {
            if (s == kSlices / 2) v = (int)(V - ((long long)vh << 28));
            const int p = kSliceBits * (kSlices / 2 - 1 - s % (kSlices / 2));   // 21, 14, 7, 0
            const int q = p ? (v + (1 << (p - 1))) >> p : v;    // nearest, ties up
            v -= q << p;                                        // |v| <= 2^(p - 1)
            t[s][kk][rr] = __float2bfloat16_rn((float)q);       // |q| <= 128: exact
        }
    }
    __syncthreads();
    // 16-byte pieces: 8 consecutive K of one row and slice
    const int nkc = kpad / kKC;
    uint8_t *ob = reinterpret_cast<uint8_t *>(left ? outa : outb);
    for (int idx = threadIdx.x; idx < kSlices * 64 * 4; idx += kThr) {
        const int rr = idx & 63, k8 = (idx >> 6) & 3, s = idx >> 8;
        const int r = r0 + rr, kk = k0 + 8 * k8;
        __align__(16) __nv_bfloat16 w[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) w[q] = t[s][8 * k8 + q][rr];
        const size_t blk = ((size_t)(r / tr) * nkc + kk / kKC) * kSlices + s;
        const uint32_t off = tc::kmajor_offset(r % tr, (kk % kKC) * 2, kKBytes);
        *reinterpret_cast<uint4 *>(ob + blk * (size_t)tr * kKBytes + off) = *reinterpret_cast<const uint4 *>(w);
    }
}

// hi 2^-21 + lo 2^-49 (|hi|, |lo| < 2^47) rounded to FP64, on integers (the FP64
// pipe, two lanes a clock, held a quarter of the kernel with conversions and
// multiply-adds): the sum as a 28 + 48 bit number, its leading 53 bits rounded.
// 1024 x 4096 outputs, 2J = 512, 550 and 1024: 231, 290, 408 -> 214, 255, 374 us.
__device__ __forceinline__ double join_levels(long long hi, long long lo) {
    constexpr unsigned int kLow = (1u << 28) - 1;
    const long long s = hi + (lo >> 28);
    const unsigned int r = (unsigned int)lo & kLow;
    const bool neg = s < 0;
    const unsigned long long a = neg ? (unsigned long long)(-s - (r != 0u)) : (unsigned long long)s;
    const unsigned long long b = neg ? (0u - r) & kLow : r;
    if (a == 0ull) return fma((double)hi, 0x1p-21, (double)lo * 0x1p-49);
    const int c = __clzll((long long)a);   // 15 .. 63
    const unsigned long long y = (a << c) | (c >= 28 ? b << (c - 28) : b >> (28 - c));
    const unsigned long long m = (y >> 11) + ((y >> 10) & 1ull);   // 2^52 .. 2^53
    const unsigned long long e = (unsigned long long)(neg ? 2048 + 1064 - c : 1064 - c);
    return __longlong_as_double((long long)((e << 52) + m));
}

// v 2^k
__device__ __forceinline__ double scale_pow2(double v, int k) {
    if (k > 1000 || k < -1000) return ldexp(v, k);
    return v * __hiloint2double((k + 1023) << 20, 0);
}

__global__ void __launch_bounds__(kCtaThreads, 1) contract_tc_kernel(
    const uint8_t *__restrict__ As, const uint8_t *__restrict__ Bs, int kpad, const int *__restrict__ ea,
    const int *__restrict__ eb, Src sa, Src sb, double *__restrict__ u, int *__restrict__ err) {
    extern __shared__ uint8_t dsm[];
    uint8_t *sm = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(dsm) + 1023) & ~(uintptr_t)1023);
    __shared__ uint64_t full[kStages], empty[kStages], lv_full, lv_empty;
    __shared__ uint32_t tslot;
    __shared__ int failed;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int x0 = blockIdx.y * kTM, t0 = blockIdx.x * kTN;
    const int nkc = kpad / kKC, nseg = (kpad + kSegK - 1) / kSegK;
    if (warp == 0) tc::tmem_alloc(&tslot, 512);
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);
        }
        tc::mbar_init(&lv_full, 1);
        tc::mbar_init(&lv_empty, 8);
        failed = 0;
    }
    tc::fence_async_smem();
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t taddr = tslot;
    double acc[2][16] = {};   // epilogue threads: sums of row 32 (warp % 4) + lane
    const uint8_t *ablk = As + (size_t)blockIdx.y * nkc * kABlock;   // this tile's chunks, in K order
    const uint8_t *bblk = Bs + (size_t)blockIdx.x * nkc * kBBlock;
    if (tid == 0) {
        // producer: chunk k's A and B blocks into stage k % kStages
        for (int k = 0; k < nkc; ++k) {
            const int st = k % kStages;
            if (k >= kStages && !tc::mbar_wait(&empty[st], (uint32_t)(((k / kStages) - 1) & 1), kWaitLimit)) {
                failed = 1;
                break;
            }
            tc::mbar_arrive_tx(&full[st], kStage);
            tc::bulk_load(sm + st * kStage, ablk + (size_t)k * kABlock, kABlock, &full[st]);
            tc::bulk_load(sm + st * kStage + kABlock, bblk + (size_t)k * kBBlock, kBBlock, &full[st]);
        }
    } else if (tid == 32) {
        // MMA issuer.  The B slices of a stage are consecutive 64-row blocks of
        // one K-major operand, so A slice i against B slices j0 .. j0 + n - 1
        // (N = 64 n <= 256) writes the products a_i b_j to accumulator columns
        // 64 (i + j): the level of each pair.  Twelve MMAs cover the 36 pairs.
        constexpr uint32_t sbo = (kKBytes / 16) * 128;
        const uint64_t desc0 = tc::smem_desc(tc::smem_u32(sm), 128, sbo);
        for (int k = 0; k < nkc && !failed; ++k) {
            const int st = k % kStages, kin = k % (kSegK / kKC);
            if (!tc::mbar_wait(&full[st], (uint32_t)((k / kStages) & 1), kWaitLimit) ||
                (kin == 0 && k > 0 && !tc::mbar_wait(&lv_empty, (uint32_t)(((k / (kSegK / kKC)) - 1) & 1), kWaitLimit))) {
                failed = 1;
                break;
            }
            tc::tc_fence_after();
            const uint64_t ds = desc0 + (uint64_t)((st * kStage) >> 4);
#pragma unroll
            for (int i = 0; i < kSlices; ++i) {
                const uint64_t da = ds + (uint64_t)((i * kASlice) >> 4);
#pragma unroll
                for (int j0 = 0; j0 < kSlices - i; j0 += 4) {
                    const int n = (kSlices - i - j0) < 4 ? (kSlices - i - j0) : 4;   // slices of B
                    const uint64_t db = ds + (uint64_t)((kABlock + j0 * kBSlice) >> 4);
                    const uint32_t id = tc::instr_desc(1u, kTM, kTN * n);
                    tc::mma<1>(taddr + (uint32_t)((i + j0) * kTN), da, db, id, (kin == 0 && i == 0) ? 0u : 1u);
                }
            }
            tc::mma_commit(&empty[st]);
            if (kin == kSegK / kKC - 1 || k == nkc - 1) tc::mma_commit(&lv_full);   // a segment's levels
        }
    } else if (warp >= 4) {
        // epilogue: warp w reads TMEM lanes 32 (w % 4) .. (rows), columns
        // 32 ((w - 4) / 4) .. of each level
        const int q = warp & 3, ch = (warp - 4) >> 2;
        bool ok = true;
        for (int sg = 0; sg < nseg && ok; ++sg) {
            ok = tc::mbar_wait(&lv_full, (uint32_t)(sg & 1), kWaitLimit);
            if (tc::bar_or(1, 256, !ok)) {   // the same verdict in every epilogue thread
                ok = false;
                break;
            }
            tc::tc_fence_after();
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                const int c0 = 32 * ch + 16 * g;
                long long hi[16], lo[16];   // levels 0 .. 3 and 4 .. 7
#pragma unroll
                for (int c = 0; c < 16; ++c) hi[c] = lo[c] = 0;
                auto join = [&](long long (&h)[16], int d0) {
#pragma unroll 1
                    for (int d = d0; d < d0 + kSlices / 2; ++d) {
                        float v[16];
                        tc::tmem_ld16(taddr + ((uint32_t)(32 * q) << 16) + (uint32_t)(d * kTN + c0), v);
#pragma unroll
                        for (int c = 0; c < 16; ++c)   // below 2^47 in magnitude
                            h[c] = h[c] * (1 << kSliceBits) + __float2int_rn(v[c]);
                    }
                };
                join(hi, 0);
                join(lo, kSlices / 2);
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    const double v = join_levels(hi[c], lo[c]);
                    acc[g][c] = sg == 0 ? v : acc[g][c] + v;
                }
            }
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&lv_empty);   // the levels may be overwritten
        }
        if ((!ok || kTestGivesUp) && lane == 0) failed = 1;
    }
    // drain: loads and MMAs in flight have landed before the CTA ends (a
    // no-op unless a wait gave up)
    if (tid == 0) {
        for (int k = max(0, nkc - kStages); k < nkc; ++k)
            tc::mbar_wait(&full[k % kStages], (uint32_t)((k / kStages) & 1), kWaitLimit);
    } else if (tid == 32) {
        for (int k = max(0, nkc - kStages); k < nkc; ++k)
            tc::mbar_wait(&empty[k % kStages], (uint32_t)((k / kStages) & 1), kWaitLimit);
    }
    tc::tc_fence_before();
    __syncthreads();
    if (failed && err && tid == 0) atomicOr(err, 1);
    if (warp >= 4) {
        // through shared memory (the stages are idle now), so that rows are
        // stored 256 bytes at a time
        const int q = warp & 3, ch = (warp - 4) >> 2;
        double *tile = reinterpret_cast<double *>(sm) + (warp - 4) * 32 * kOutPitch;
#pragma unroll
        for (int g = 0; g < 2; ++g)
#pragma unroll
            for (int c = 0; c < 16; ++c) tile[lane * kOutPitch + 16 * g + c] = acc[g][c];
        __syncwarp();
        const int t = t0 + 32 * ch + lane, J = sa.J, n_x = sa.rows, n_T = sb.rows;
        const int et = eb[t], rows = min(32, n_x - (x0 + 32 * q));
        if (t < n_T)
            for (int r = 0; r < rows; ++r) {
                const int x = x0 + 32 * q + r, ex = ea[x];
                double v;
                if (failed || ex == kNonFinite || et == kNonFinite) {
                    v = 0.0;
                    for (int j = 0; j < J; ++j) v = fma(sa.V[(long long)j * n_x + x].x, sb.G0[(long long)j * n_T + t], v);
                    for (int j = 0; j < J; ++j) v = fma(sa.V[(long long)j * n_x + x].y, sb.G1[(long long)j * n_T + t], v);
                } else {
                    v = scale_pow2(tile[r * kOutPitch + lane], ex + et - 2 * kSliceBits);
                }
                u[(long long)x * n_T + t] = v;
            }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_free(taddr, 512);
}

}  // namespace

int contract_tc_kpad(int J) { return (2 * J + kKPad - 1) / kKPad * kKPad; }
int contract_tc_rows(int n) { return (n + kTM - 1) / kTM * kTM; }
int contract_tc_cols(int n) { return (n + kTN - 1) / kTN * kTN; }
bool contract_tc_ok(int J) { return 2 * J <= kContractTcMaxK; }

size_t contract_tc_scratch_bytes(int J, int n_x, int n_T) {
    const size_t kp = (size_t)contract_tc_kpad(J);
    const size_t rx = (size_t)contract_tc_rows(n_x), rt = (size_t)contract_tc_cols(n_T);
    return (size_t)kSlices * (rx + rt) * kp * sizeof(__nv_bfloat16) + (rx + rt + kp) * sizeof(int);
}

cudaError_t launch_contract_tc(int J, int n_x, int n_T, const double2 *V, const double *Gr,
                               const double *Gm, double *u, void *scratch, int *err, cudaStream_t st) {
    if (n_x <= 0 || n_T <= 0) return cudaSuccess;
    static std::atomic<unsigned long long> attr{0};
    {
        const cudaError_t e = ensure_smem_attr((const void *)contract_tc_kernel, kSmem, attr);
        if (e != cudaSuccess) return e;
    }
    const int kp = contract_tc_kpad(J), rx = contract_tc_rows(n_x), rt = contract_tc_cols(n_T);
    __nv_bfloat16 *As = static_cast<__nv_bfloat16 *>(scratch);
    __nv_bfloat16 *Bs = As + (size_t)kSlices * rx * kp;
    int *ea = reinterpret_cast<int *>(Bs + (size_t)kSlices * rt * kp);
    int *eb = ea + rx, *d = eb + rt;
    const Src sa{V, nullptr, nullptr, J, n_x}, sb{nullptr, Gr, Gm, J, n_T};
    ozaki_scale_kernel<<<(rx + rt) / 32, kScaleThr, 0, st>>>(sa, sb, rx / 32, nullptr, ea, eb);
    ozaki_balance_kernel<<<J, kThr, 0, st>>>(sa, sb, ea, eb, d);
    ozaki_scale_kernel<<<(rx + rt) / 32, kScaleThr, 0, st>>>(sa, sb, rx / 32, d, ea, eb);
    ozaki_slice_kernel<<<dim3((rx + rt) / 64, kp / 32), kThr, 0, st>>>(sa, sb, rx / 64, d, ea, eb, kp, As, Bs);
    contract_tc_kernel<<<dim3(rt / kTN, rx / kTM), kCtaThreads, kSmem, st>>>(
        reinterpret_cast<const uint8_t *>(As), reinterpret_cast<const uint8_t *>(Bs), kp, ea, eb, sa, sb, u, err);
    return cudaGetLastError();
}

}  // namespace fh
