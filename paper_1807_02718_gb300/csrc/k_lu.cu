// Step a3: batched dense complex LU with partial pivoting and the solve
// A_s psi_s = g_s for every frequency (Sec. 5 step F3; the paper solves its 2D
// systems directly and notes LU for small problems in its appendix).
//
// FP64 path: right-looking blocked LU (panels of NB = 16 columns) on the
// column-major matrices, all systems advancing together.  The right side is
// carried as column N, so that row exchanges and eliminations reach it in
// flight; L is not needed once its panel's update is done, so columns left of
// a panel are never exchanged.  Per panel two launches over the systems that
// still have one (a prefix of the order, largest first):
//   panel  one CTA per system: partial pivoting within the panel;
//   strip  one CTA per SW columns right of it: the panel's row exchanges, U12
//          = L11^{-1} A12, then A22 -= L21 U12 for all rows of the strip.
// Every second system runs on a second stream, so that one half's panels
// (short dependent steps that leave most of the chip idle) overlap with the
// other half's strips.
//
// Bound: the FP64 pipe, two FMAs per clock and SM (1.25 TFLOP/s measured), so
// that one warp's FMA occupies an SM for 16 clocks: loads, shared memory and
// launches are nearly free, and what counts is that every SM has FMAs to
// issue.  One CTA per system, as before, leaves the largest system on one SM
// (N = 480: 36 ms at the SM's peak) and 63 systems on 63 SMs; strips of SW = 8
// columns spread each system over N / 8 CTAs.
// Measured (GB300, LU phase; the flops at peak take 2.3 and 17 ms): 63 systems
// of N = 256: 14.3 -> 3.5 ms; 255 systems of N = 64..480: 78.0 -> 20.5 ms
// (strips of 16 columns: 3.8 and 21.1 ms).
#include <algorithm>

#include "fh_internal.h"

namespace fh {
namespace {

constexpr int NB = 16;             // panel width
constexpr int kPanelRows = 512;    // panels of at most this many rows stay in registers
constexpr int SW = 8;              // columns of a strip
constexpr int kStripThreads = 128;
constexpr int kMaxMoved = 2 * NB;

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cinv(double2 a) {
    const double d = a.x * a.x + a.y * a.y;
    return make_double2(a.x / d, -a.y / d);
}
// v -= l u in four FMAs (as v -= (l.x u.x - l.y u.y) it takes six instructions)
__device__ __forceinline__ void csub(double2 &v, double2 l, double2 u) {
    v.x = fma(l.y, u.y, fma(-l.x, u.x, v.x));
    v.y = fma(-l.y, u.x, fma(-l.x, u.y, v.y));
}

// Rows that a panel moves, relative to its first row: row src goes to dst.
struct Moves {
    int cnt, dst[kMaxMoved], src[kMaxMoved];
};

// Pivot key of an active row: the bits of |re| + |im| (monotone as integers;
// NaN above everything), then ~position (the smaller position wins a tie).
struct Key {
    unsigned hi, lo, pos;
};
__device__ __forceinline__ Key key_of(double2 v, int pos) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(fabs(v.x) + fabs(v.y));
    return {(unsigned)(b >> 32), (unsigned)b, ~(unsigned)pos};
}
__device__ __forceinline__ Key warp_max(Key k) {
    const unsigned h = __reduce_max_sync(0xffffffffu, k.hi);
    const unsigned l = __reduce_max_sync(0xffffffffu, k.hi == h ? k.lo : 0u);
    const unsigned p = __reduce_max_sync(0xffffffffu, k.hi == h && k.lo == l ? k.pos : 0u);
    return {h, l, p};
}
__device__ __forceinline__ bool key_less(Key a, Key b) {
    return a.hi != b.hi ? a.hi < b.hi : a.lo != b.lo ? a.lo < b.lo : a.pos < b.pos;
}
__device__ __forceinline__ bool key_bad(Key k) {   // nothing left, zero, infinite or NaN
    return k.pos == 0u || (k.hi | k.lo) == 0u || k.hi >= 0x7FF00000u;
}

struct PanelShared {
    Key best[2][kPanelRows / 32];   // best key of every warp
    double2 row[2][NB];             // the pivot row from its column on
    double2 pinv[2];
    Moves mv;
};

// Columns k0 .. k0 + 15 of system order[first + 2 blockIdx.x]: up to 512 rows
// with one row per thread in registers.  Rows do not move; each thread tracks
// the position its row has under the exchanges, and rows go to their final
// place at the end.  Per column: keys reduced by redux within the warps and
// across them, the winning thread publishes its row and the reciprocal of the
// pivot (one division per column: a warp's FP64 division occupies the SM's
// pipe for ~500 clocks), the others eliminate.
__device__ void panel_registers(double2 *a, int n, int k0, PanelShared &ps, int *info) {
    const int m = n - k0, nb = min(NB, m), t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int nw = blockDim.x >> 5;
    double2 v[NB];
    const bool own = t < m;
#pragma unroll
    for (int q = 0; q < NB; ++q)
        v[q] = own && q < nb ? a[(long long)(k0 + q) * n + k0 + t] : make_double2(0.0, 0.0);
    int pos = t;
    bool active = own;
#pragma unroll
    for (int c = 0; c < NB; ++c) {
        if (c >= nb) break;
        const int pb = c & 1;
        const Key mine = active ? key_of(v[c], pos) : Key{0u, 0u, 0u};
        const Key wb = warp_max(mine);
        if (lane == 0) ps.best[pb][warp] = wb;
        __syncthreads();
        const Key k = warp_max(lane < nw ? ps.best[pb][lane] : Key{0u, 0u, 0u});
        if (key_bad(k)) {   // the same verdict in every thread
            if (t == 0) *info = k0 + c + 1;
            return;
        }
        const int wpos = (int)~k.pos;
        if (active && pos == wpos) {
#pragma unroll
            for (int q = c; q < NB; ++q) ps.row[pb][q] = v[q];
            ps.pinv[pb] = cinv(v[c]);
            pos = c;
            active = false;
        } else if (active && pos == c) {
            pos = wpos;   // exchanged with the pivot row
        }
        __syncthreads();
        if (active) {
            const double2 l = cmul(v[c], ps.pinv[pb]);
            v[c] = l;
#pragma unroll
            for (int q = c + 1; q < NB; ++q) csub(v[q], l, ps.row[pb][q]);
        }
    }
    if (own) {
#pragma unroll
        for (int q = 0; q < NB; ++q)
            if (q < nb) a[(long long)(k0 + q) * n + k0 + pos] = v[q];
        if (pos != t) {
            const int i = atomicAdd(&ps.mv.cnt, 1);
            if (i < kMaxMoved) {   // at most 2 NB rows change position
                ps.mv.dst[i] = pos;
                ps.mv.src[i] = t;
            }
        }
    }
}

// The same panel for any number of rows, in place: rows are exchanged in the
// panel's columns; the update of a column's right neighbours also finds the
// next column's best key.
__device__ void panel_memory(double2 *a, int n, int k0, PanelShared &ps, int *info) {
    const int m = n - k0, nb = min(NB, m), t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int nw = blockDim.x >> 5;
    double2 *p0 = a + (long long)k0 * n + k0;   // panel element (r, q) at p0[q n + r]
    Key next = {0u, 0u, 0u};
    for (int r = t; r < m; r += blockDim.x) {
        const Key k = key_of(p0[r], r);
        if (key_less(next, k)) next = k;
    }
    for (int c = 0; c < nb; ++c) {
        const int pb = c & 1;
        const Key wb = warp_max(next);
        if (lane == 0) ps.best[pb][warp] = wb;
        __syncthreads();
        const Key k = warp_max(lane < nw ? ps.best[pb][lane] : Key{0u, 0u, 0u});
        if (key_bad(k)) {
            if (t == 0) *info = k0 + c + 1;
            return;
        }
        const int wpos = (int)~k.pos;
        if (t < nb) {
            double2 *col = p0 + (long long)t * n;
            const double2 u = col[wpos];
            if (wpos != c) {
                col[wpos] = col[c];
                col[c] = u;
            }
            ps.row[pb][t] = u;
            if (t == c) ps.pinv[pb] = cinv(u);
        }
        if (t == 0 && wpos != c) {   // compose the exchange (c, wpos) with the moves so far
            int ic = -1, ip = -1;
            for (int i = 0; i < ps.mv.cnt; ++i) {
                if (ps.mv.dst[i] == c) ic = i;
                if (ps.mv.dst[i] == wpos) ip = i;
            }
            if (ic < 0) {
                ic = ps.mv.cnt++;
                ps.mv.dst[ic] = ps.mv.src[ic] = c;
            }
            if (ip < 0) {
                ip = ps.mv.cnt++;
                ps.mv.dst[ip] = ps.mv.src[ip] = wpos;
            }
            const int s0 = ps.mv.src[ic];
            ps.mv.src[ic] = ps.mv.src[ip];
            ps.mv.src[ip] = s0;
        }
        __syncthreads();
        const double2 pinv = ps.pinv[pb];
        next = {0u, 0u, 0u};
        for (int r = c + 1 + t; r < m; r += blockDim.x) {
            const double2 l = cmul(p0[(long long)c * n + r], pinv);
            p0[(long long)c * n + r] = l;
            for (int q = c + 1; q < nb; ++q) {
                double2 v = p0[(long long)q * n + r];
                csub(v, l, ps.row[pb][q]);
                p0[(long long)q * n + r] = v;
                if (q == c + 1) {
                    const Key k1 = key_of(v, r);
                    if (key_less(next, k1)) next = k1;
                }
            }
        }
    }
}

__global__ void __launch_bounds__(kPanelRows) lu_panel_fp64_kernel(
    const int *__restrict__ order, const int *__restrict__ Ns, const long long *__restrict__ mat_off,
    double2 *__restrict__ A, Moves *__restrict__ moves, int *__restrict__ info, int k0) {
    __shared__ PanelShared ps;
    const int s = order[2 * blockIdx.x];
    if (info[s] != 0) return;
    const int n = Ns[s];
    double2 *a = A + mat_off[s];
    if (threadIdx.x == 0) ps.mv.cnt = 0;
    __syncthreads();
    // by the system's own size, so that its result does not depend on the batch
    if (n - k0 <= kPanelRows) panel_registers(a, n, k0, ps, info + s);
    else panel_memory(a, n, k0, ps, info + s);
    __syncthreads();
    Moves *mv = moves + s;
    for (int i = threadIdx.x; i < kMaxMoved; i += blockDim.x) {
        mv->dst[i] = ps.mv.dst[i];
        mv->src[i] = ps.mv.src[i];
    }
    if (threadIdx.x == 0) mv->cnt = min(ps.mv.cnt, kMaxMoved);
}

// Columns j0 .. j0 + SW - 1 (j0 = k0 + 16 + SW blockIdx.x; column n is the right
// side) of system order[first + 2 blockIdx.y]: exchanges, U12, update.  A
// thread takes a row with its 16 values of L in registers; U12 is broadcast
// from shared memory (one 16-byte read per four FMAs).
__global__ void __launch_bounds__(kStripThreads, 4) lu_strip_fp64_kernel(
    const int *__restrict__ order, const int *__restrict__ Ns, const long long *__restrict__ mat_off,
    const int *__restrict__ vec_off, double2 *__restrict__ A, double2 *__restrict__ B,
    const Moves *__restrict__ moves, const int *__restrict__ info, int k0) {
    __shared__ double2 L11[NB][NB + 1], U[SW][NB];   // U[column][row]
    const int s = order[2 * blockIdx.y], n = Ns[s];
    const int nb = min(NB, n - k0), j0 = k0 + nb + SW * (int)blockIdx.x;
    if (j0 > n || info[s] != 0) return;
    const int nc = min(SW, n + 1 - j0), t = threadIdx.x;
    double2 *a = A + mat_off[s], *y = B + vec_off[s];
    auto column = [&](int j) { return j < n ? a + (long long)j * n : y; };
    // row exchanges: every moved row of the strip is read before any is written
    const int nmv = moves[s].cnt;
    double2 mvv[kMaxMoved * SW / kStripThreads];
#pragma unroll
    for (int i = 0; i < kMaxMoved * SW / kStripThreads; ++i) {
        const int e = t + i * kStripThreads, p = e & (kMaxMoved - 1), c = e / kMaxMoved;
        if (p < nmv && c < nc) mvv[i] = column(j0 + c)[k0 + moves[s].src[p]];
    }
    for (int e = t; e < NB * NB; e += kStripThreads) {
        const int r = e % NB, q = e / NB;
        L11[r][q] = r < nb && q < r ? a[(long long)(k0 + q) * n + k0 + r] : make_double2(0.0, 0.0);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kMaxMoved * SW / kStripThreads; ++i) {
        const int e = t + i * kStripThreads, p = e & (kMaxMoved - 1), c = e / kMaxMoved;
        if (p < nmv && c < nc) column(j0 + c)[k0 + moves[s].dst[p]] = mvv[i];
    }
    __syncthreads();
    // U12: half a warp per column, lane r holds row r
    const int r = t & (NB - 1);
#pragma unroll
    for (int h = 0; h < NB * SW / kStripThreads; ++h) {
        const int c = t / NB + h * (kStripThreads / NB);
        double2 *col = column(j0 + min(c, nc - 1)) + k0;
        double2 x = r < nb ? col[r] : make_double2(0.0, 0.0);
#pragma unroll
        for (int q = 0; q < NB - 1; ++q) {
            const double2 xq = make_double2(__shfl_sync(0xffffffffu, x.x, q, NB), __shfl_sync(0xffffffffu, x.y, q, NB));
            if (r > q) csub(x, L11[r][q], xq);
        }
        if (c < nc && r < nb) col[r] = x;
        U[c][r] = x;
    }
    __syncthreads();
    const int r0 = k0 + nb;   // nb == NB whenever rows are left
    for (int i = r0 + t; i < n; i += kStripThreads) {
        double2 l[NB];
#pragma unroll
        for (int q = 0; q < NB; ++q) l[q] = a[(long long)(k0 + q) * n + i];
#pragma unroll 2
        for (int c = 0; c < nc; ++c) {
            double2 *p = column(j0 + c) + i;
            double2 v = *p;
#pragma unroll
            for (int q = 0; q < NB; ++q) csub(v, l[q], U[c][q]);
            *p = v;
        }
    }
}

// Back substitution U x = y in place, one CTA per system, blocks of 16
// columns from the last: half a warp solves the diagonal block (lane r holds
// row r), then every row above subtracts the block's 16 products.
__global__ void __launch_bounds__(256) lu_back_fp64_kernel(
    const int *__restrict__ order, const int *__restrict__ Ns, const long long *__restrict__ mat_off,
    const int *__restrict__ vec_off, const double2 *__restrict__ A, double2 *__restrict__ B,
    const int *__restrict__ info) {
    __shared__ double2 xs[NB];
    const int s = order[blockIdx.x], n = Ns[s], t = threadIdx.x;
    if (info[s] != 0) return;
    const double2 *a = A + mat_off[s];
    double2 *y = B + vec_off[s];
    for (int jb = (n - 1) / NB * NB; jb >= 0; jb -= NB) {
        const int nb = min(NB, n - jb);
        if (t < NB) {
            double2 u[NB];
#pragma unroll
            for (int q = 0; q < NB; ++q)
                u[q] = t < nb && q >= t && q < nb ? a[(long long)(jb + q) * n + jb + t] : make_double2(0.0, 0.0);
            double2 x = t < nb ? y[jb + t] : make_double2(0.0, 0.0);
            double2 inv = make_double2(0.0, 0.0);   // reciprocal of the lane's diagonal entry
#pragma unroll
            for (int q = 0; q < NB; ++q)
                if (q == t) inv = u[q];
            inv = t < nb ? cinv(inv) : inv;
#pragma unroll
            for (int q = NB - 1; q >= 0; --q) {
                if (t == q) x = cmul(x, inv);
                const double2 xq = make_double2(__shfl_sync(0xffffu, x.x, q, NB), __shfl_sync(0xffffu, x.y, q, NB));
                if (t < q && q < nb) csub(x, u[q], xq);
            }
            if (t < nb) y[jb + t] = x;
            xs[t] = x;
        }
        __syncthreads();
        for (int i = t; i < jb; i += blockDim.x) {
            double2 v = y[i];
#pragma unroll
            for (int q = NB - 1; q >= 0; --q)
                if (q < nb) csub(v, a[(long long)(jb + q) * n + i], xs[q]);
            y[i] = v;
        }
        __syncthreads();
    }
}

}  // namespace

size_t lu_fp64_scratch_bytes(int S) { return (size_t)S * sizeof(Moves); }

int lu_fp64_launches(const int *order_h, const int *N_h, int S) {
    int n = S > 0 ? 1 : 0;
    for (int half = 0; half < 2 && half < S; ++half) n += 2 * ((N_h[order_h[half]] + NB - 1) / NB);
    return n;
}

void launch_lu_solve_fp64(const int *order, const int *order_h, const int *N_h, int S, const int *N,
                          const long long *mat_off, const int *vec_off, double2 *A, double2 *b, int *info,
                          void *scratch, cudaStream_t st, cudaStream_t side, cudaEvent_t fork, cudaEvent_t join) {
    if (S <= 0) return;
    Moves *mv = static_cast<Moves *>(scratch);
    cudaEventRecord(fork, st);
    cudaStreamWaitEvent(side, fork, 0);
    for (int half = 0; half < 2 && half < S; ++half) {   // systems half, half + 2, .. of the order
        cudaStream_t q = half ? side : st;
        int active = (S - half + 1) / 2;
        const int n0 = N_h[order_h[half]];
        for (int k0 = 0; k0 < n0; k0 += NB) {
            while (N_h[order_h[half + 2 * (active - 1)]] <= k0) --active;
            const int rows = std::min(n0 - k0, kPanelRows);
            lu_panel_fp64_kernel<<<active, (rows + 31) / 32 * 32, 0, q>>>(order + half, N, mat_off, A, mv, info, k0);
            // columns right of the panel with the right side (the smaller systems' extra CTAs return)
            const int strips = (std::max(n0 - k0 - NB, 0) + SW) / SW;
            lu_strip_fp64_kernel<<<dim3(strips, active), kStripThreads, 0, q>>>(order + half, N, mat_off, vec_off, A,
                                                                                b, mv, info, k0);
        }
    }
    cudaEventRecord(join, side);
    cudaStreamWaitEvent(st, join, 0);
    lu_back_fp64_kernel<<<S, 256, 0, st>>>(order, N, mat_off, vec_off, A, b, info);
}

}  // namespace fh
