// tl_smem.cuh -- LUpp with the matrices in shared memory, T lanes per
// system, run-time n (<= 32).
//
// Each system is an augmented n x (n+1) row-major block in shared memory
// (column n holds b, then y, then x), rows RS doubles apart (RS odd), then
// n reciprocals and n pivot rows.  The interchanges of Sec. 2.2 swap whole
// rows in place, the T lanes sharing the columns.
//
// Two eliminations share this layout:
//   * smem_lupp2 (the fast path): the trailing block is walked element by
//     element, lane t taking every T-th element row-major, and the updates
//     of two elimination steps are applied in one pass; see its comment.
//   * smem_lupp: one step per pass on a TR x TC tile of lanes (lane (tr, tc)
//     keeps its columns of the pivot row in registers and walks its rows);
//     2, 4 or 8 lanes, kept for the lane-tile variants.
// The kernels: k_smem_group (fixed-size batches, both layouts, loads into
// shared memory by cp.async) and k_smem_ragged (one size of a ragged batch,
// the per-size mode).
//
// Arithmetic is the same as the register solvers of tinylu_device.cuh (negated
// multipliers a_ik * (-RN(1/a_kk)), one FMA per update in increasing k, the
// back substitution by RN(1/u_ii)); LU and pivots are bit-identical to the
// sequential elimination.
#pragma once
#include "tinylu.h"
#include "tl_bounds.cuh"
#include "tl_kernels.cuh"

// Unroll factor of the row loop of the lane-tile trailing update (2
// measured 5-10% slower than 1).
#ifndef TL_SMEM_ROW_UNROLL
#define TL_SMEM_ROW_UNROLL 1
#endif

namespace tl {

constexpr int kSmemRowUnroll = TL_SMEM_ROW_UNROLL;

// Row stride of a system's n x (n+1) block: the smallest odd number of
// doubles >= n+1, so that a column walked by consecutive lanes hits distinct
// banks and the block stays small (shared memory bounds the warps resident
// per SM).
__host__ __device__ constexpr int smem_row_stride(int n) { return (n + 1) | 1; }

// Offsets (in doubles) of the n reciprocals RN(1/u_kk) and of the n pivot
// rows (int32, two per double) behind a system's n x RS block.
__host__ __device__ constexpr int smem_rcp_offset(int n) { return n * smem_row_stride(n); }
__host__ __device__ constexpr int smem_piv_offset(int n) { return n * smem_row_stride(n) + n; }

// Shared-memory footprint of one system in doubles: the n x RS block, n
// reciprocals, n pivots.  Padded so that consecutive systems start T slots
// apart modulo 16 (the systems of one half-warp then do not collide on a
// bank).
__host__ __device__ constexpr int smem_sys_doubles(int n, int T = 16)
{
    const int base = smem_piv_offset(n) + (n + 1) / 2;
    const int want = T < 16 ? T : T / 8;
    return base + ((want - base % 16) % 16 + 16) % 16;
}
__host__ __device__ constexpr size_t smem_sys_bytes(int n, int T = 16)
{
    return static_cast<size_t>(smem_sys_doubles(n, T)) * 8;
}

template <int T>
__device__ __forceinline__ int group_any_int(int v)
{
#pragma unroll
    for (int off = T / 2; off >= 1; off >>= 1) v |= __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// Elimination of one system held by the T lanes of a group: the augmented
// n x (n+1) block M (row stride RS; column n = b when SOLVE), followed by
// n reciprocals and n pivot rows.  LUpp with the arithmetic of the
// register solvers (negated multipliers a_ik * (-RN(1/a_kk)), one FMA per
// update in increasing k, b carried as column n, back substitution by
// RN(1/u_ii)); on return M holds L (negated, below the diagonal) and U, and
// column n holds x when SOLVE.  Returns info.  Every lane of the warp must
// call it together (shuffles and votes inside).
//
// Trailing updates on a TR x TC tile of lanes: lane (tr, tc) updates rows
// k+1+tr, k+1+tr+TR, ... and columns k+1+tc, k+1+tc+TC, ..., keeping its
// columns of the pivot row in registers.
template <int T, bool SOLVE>
__device__ __forceinline__ int smem_lupp(double *M, int n, int RS, int t, int tile, double threshold)
{
    constexpr int MODE = SOLVE ? kGesv : kGetrf;
    constexpr int TC = T >= 4 ? 4 : T;  // lane tile
    constexpr int TR = T / TC;
    constexpr int MAXC = TL_MAX_N / TC;  // whole column chunks per lane (at most 32 live columns)
    static_assert(MAXC <= 16, "the chunk switch below covers 16 chunks");
    static_assert(T >= 1 && T <= 32 && (32 % T) == 0, "T must divide 32");
    const int tr = t / TC, tc = t % TC;
    double *rcp = M + n * RS;                              // n doubles
    int *piv = reinterpret_cast<int *>(rcp + n);           // n ints
    int info = 0;
    bool tiny = false;
    const int wcols = n + (MODE == kGesv ? 1 : 0);         // columns incl. b
    for (int k = 0; k < n; ++k) {
        // a2: first maximum of |a_ik| over rows k..hi-1: the whole column,
        // or with tile-local pivoting the diagonal tile first and the rows
        // below it only when the tile's best magnitude is under the
        // threshold (the first maximum over k..n-1 then)
        int hi = n;
        if (tile > 0 && tile < n) hi = min(n, (k / tile + 1) * tile);
        double cv = 0.0;
        int cpos = n;
        for (int i = k + t; i < hi; i += T) {
            const double v = M[i * RS + k];
            if (cpos == n || dev::mag_bits(v) > dev::mag_bits(cv)) { cv = v; cpos = i; }
        }
        dev::group_argmax<T>(cv, cpos);
        if (hi < n) {
            const bool below = dev::mag_bits(cv) < dev::mag_bits(threshold);
            if (below) {
                for (int i = hi + ((t - hi) % T + T) % T; i < n; i += T) {
                    const double v = M[i * RS + k];
                    if (dev::mag_bits(v) > dev::mag_bits(cv)) { cv = v; cpos = i; }
                }
            }
            if (__any_sync(0xffffffffu, below)) dev::group_argmax<T>(cv, cpos);
        }
        const int p = cpos;
        const bool zero = dev::mag_bits(cv) == 0ULL;
        if (zero && info == 0) info = k + 1;
        if (t == 0) piv[k] = p;
        // a3: physical interchange of rows k and p (L part and b included)
        if (p != k) {
            for (int j = t; j < wcols; j += T) {
                const double tmp = M[k * RS + j];
                M[k * RS + j] = M[p * RS + j];
                M[p * RS + j] = tmp;
            }
        }
        __syncwarp();
        // a4: reciprocal and negated multipliers
        const bool small = !zero && dev::mag_bits(cv) < dev::kDblMinBits;
        const double r = dev::rcp_rn(cv);
        if (t == 0) rcp[k] = r;
        tiny = tiny || small;
        const double nr = dev::neg(r);
        if (!__any_sync(0xffffffffu, small)) {
            for (int i = k + 1 + t; i < n; i += T) {
                double *a = &M[i * RS + k];
                *a = zero ? dev::neg(*a) : __dmul_rn(*a, nr);
            }
        } else {
            const double ncv = dev::neg(cv);
            for (int i = k + 1 + t; i < n; i += T) {
                double *a = &M[i * RS + k];
                *a = zero ? dev::neg(*a) : (small ? __ddiv_rn(*a, ncv) : __dmul_rn(*a, nr));
            }
        }
        __syncwarp();
        // a5 (+ forward part of a6 through column n): a_ij += (-l_ik) u_kj.
        if (!zero) {
            // lane (tr, tc) owns columns k+1+tc + c*TC: nfull whole chunks
            // (the same count on every lane of the warp) and possibly one
            // tail column; the chunks are a straight-line fall-through block
            // entered once per row, with immediate offsets from the row
            // pointer
            const int ncols = wcols - (k + 1);
            const int nfull = ncols / TC;
            const bool has_tail = tc < ncols - nfull * TC;
            const double *urow = M + k * RS + k + 1 + tc;
            double u[MAXC];
#pragma unroll
            for (int c = 0; c < MAXC; ++c) u[c] = c < nfull ? urow[c * TC] : 0.0;
            const double ut = has_tail ? urow[nfull * TC] : 0.0;
#pragma unroll kSmemRowUnroll
            for (int i = k + 1 + tr; i < n; i += TR) {
                double *Mi = M + i * RS;
                const double l = Mi[k];
                double *Mr = Mi + k + 1 + tc;
                switch (nfull) {
#define TL_SMEM_CHUNK(c)                                                                \
    case (c) + 1:                                                                       \
        if ((c) < MAXC) Mr[(c) * TC] = __fma_rn(l, u[(c) < MAXC ? (c) : 0], Mr[(c) * TC]); \
        [[fallthrough]];
                    TL_SMEM_CHUNK(15)
                    TL_SMEM_CHUNK(14)
                    TL_SMEM_CHUNK(13)
                    TL_SMEM_CHUNK(12)
                    TL_SMEM_CHUNK(11)
                    TL_SMEM_CHUNK(10)
                    TL_SMEM_CHUNK(9)
                    TL_SMEM_CHUNK(8)
                    TL_SMEM_CHUNK(7)
                    TL_SMEM_CHUNK(6)
                    TL_SMEM_CHUNK(5)
                    TL_SMEM_CHUNK(4)
                    TL_SMEM_CHUNK(3)
                    TL_SMEM_CHUNK(2)
                    TL_SMEM_CHUNK(1)
                    TL_SMEM_CHUNK(0)
#undef TL_SMEM_CHUNK
                default: break;
                }
                if (has_tail) Mr[nfull * TC] = __fma_rn(l, ut, Mr[nfull * TC]);
            }
        }
        __syncwarp();
    }

    // a6 (back part): x_i = y_i * RN(1/u_ii), then y_r -= u_ri x_i for r < i
    if (MODE == kGesv) {
        const bool any_tiny = __any_sync(0xffffffffu, tiny);
        for (int i = n - 1; i >= 0; --i) {
            if (t == 0) {
                const double y = M[i * RS + n];
                double xi;
                if (!any_tiny) xi = __dmul_rn(y, rcp[i]);
                else xi = tiny ? __ddiv_rn(y, M[i * RS + i]) : __dmul_rn(y, rcp[i]);
                M[i * RS + n] = xi;
            }
            __syncwarp();
            const double nxi = dev::neg(M[i * RS + n]);
            for (int r2 = t; r2 < i; r2 += T) M[r2 * RS + n] = __fma_rn(M[r2 * RS + i], nxi, M[r2 * RS + n]);
            __syncwarp();
        }
    }
    return info;
}

// ---------------------------------------------------------------------------
// Element-walk elimination with the trailing update of two steps per pass.
//
// Same result as smem_lupp bit for bit (every element still receives
// fma(-l_ik, u_kj, a_ij) in increasing k with the same operands).
// Bound by the FP64 pipe (64 clocks of a sub-partition per warp instruction,
// full or not) and, in between, by the latency of each step's serial part:
// the pivot search, the reciprocal, the interchange and the multipliers took
// 43,000 of the 73,000 clocks that a warp alone on an SM needed for four
// systems of n = 19, against 24,600 of FP64 instructions, too much for the
// three or four warps per sub-partition to hide.  So:
//   * steps k and k+1 are paired: after the pivot of step k (search, row
//     interchange, multipliers, column k+1 updated in the same pass), the
//     pivot of step k+1 is found among the values that pass just formed, the
//     row that becomes row k+1 receives its step-k update during its
//     interchange and column k+1 its multipliers; then one walk over the
//     block below and to the right of (k+1, k+1) applies both steps' updates
//     to each element (one load, two FMAs in order, one store).  Rows
//     interchanged at step k+1 still carry their pending step-k update and
//     their own -l_ik, so the interchange covers column k as well;
//   * every serial pass loads what it needs before its first arithmetic or
//     store (PivotScan, smem_swap, smem_multipliers), and passes end with
//     branches the whole warp takes: an FP64 instruction without an active
//     lane costs as much as a full one;
//   * element walk indices come from a multiply-shift instead of run-time
//     divisions;
//   * the back substitution keeps y in registers (lane t holds rows
//     t, t+T, ...) and broadcasts each x_i with a shuffle;
//   * whether A holds a non-finite entry is learned on the way (worst).
// Measured against the first form of this walk (search from shared memory by
// warp reductions, one entry at a time in every pass, a scan of A for
// non-finite entries): n = 19 per system, 313,111 systems, 0.80 -> 0.93
// TFLOP/s; n = 13 interleaved, 932,944 systems, 0.84 -> 0.89; n = 30 per
// system, 82,712 systems, 0.89 -> 0.94.
// KEEPL: interchange whole rows, L part included (getrf output); without it
// only the columns the remaining elimination reads are interchanged.
// ---------------------------------------------------------------------------

// ceil(2^16 / c): floor(x / c) == (x * kDivMagic[c]) >> 16 for 0 <= x < 64.
struct DivMagic {
    unsigned short m[65];
    constexpr DivMagic() : m()
    {
        for (int c = 1; c <= 64; ++c) m[c] = static_cast<unsigned short>((65536 + c - 1) / c == 65536 ? 0 : (65536 + c - 1) / c);
    }
};
static __constant__ const DivMagic kDivMagic{};

// floor(x / c) for 0 <= x < 64, 1 <= c <= 64.
__device__ __forceinline__ int div_small(int x, int c)
{
    return c == 1 ? x : static_cast<int>((static_cast<unsigned>(x) * kDivMagic.m[c]) >> 16);
}

// First maximum of |M[i*RS + k]| over rows i in [lo, hi) of the group's
// system: a butterfly over (magnitude, row).  Every lane of the warp together.
// The rare second stage of the pivot search, out of line.
template <int T>
static __device__ __noinline__ int smem_pivot_exact(const double *M, int RS, int k, int lo, int hi, int t, int lim)
{
    unsigned long long best = 0;
    int row = hi;
    for (int i = lo + t; i < hi; i += T) {
        const unsigned long long m = dev::mag_bits(TL_SM(M, i * RS + k, lim));
        if (row == hi || m > best) {
            best = m;
            row = i;
        }
    }
    __syncwarp();
#pragma unroll
    for (int off = T / 2; off >= 1; off >>= 1) {
        const unsigned long long ob = __shfl_xor_sync(0xffffffffu, best, off);
        const int orow = __shfl_xor_sync(0xffffffffu, row, off);
        const bool take = (orow < hi) && (row >= hi || ob > best || (ob == best && orow < row));
        best = take ? ob : best;
        row = take ? orow : row;
    }
    return row;
}

// Pivot search of one column.  Each lane proposes its candidates (add), then
// the group agrees (finish) on the largest high word of |a_ik|: log2(T)
// 32-bit shuffles (one warp reduction for T = 32), one vote, one shuffle of
// the winner.  Two candidates that share the largest high word (1e-5 of the
// columns of random systems, most columns of small integers) take the exact
// search on the whole magnitude.  On one warp per SM, n = 19 with 8 lanes:
// 470 clocks per search, 670 with a warp reduction of the high word, the low
// word and the row for each group.
struct PivotScan {
    unsigned best;  // high word of the largest magnitude + 1, 0 without a candidate
    double v;
    int row;
    bool tie;
    __device__ __forceinline__ void clear()
    {
        best = 0;
        v = 0.0;
        row = 0;
        tie = false;
    }
    __device__ __forceinline__ void add(double a, int i, bool in)
    {
        const unsigned key = in ? static_cast<unsigned>(dev::mag_bits(a) >> 32) + 1u : 0u;
        const bool gt = key > best;
        tie = gt ? false : (tie || (in && key == best));
        best = gt ? key : best;
        v = dev::sel(gt, a, v);
        row = gt ? i : row;
    }
    template <int T>
    __device__ __forceinline__ void finish(const double *M, int RS, int k, int lo, int hi, int t, int lim, double &cv,
                                           int &p) const
    {
        constexpr unsigned kMask = T == 32 ? 0xffffffffu : (1u << (T & 31)) - 1u;
        const int lane0 = (static_cast<int>(threadIdx.x) & 31) - t;
        unsigned m = best;
        if constexpr (T == 32) {
            m = __reduce_max_sync(0xffffffffu, m);
        } else {
#pragma unroll
            for (int off = T / 2; off >= 1; off >>= 1) {
                const unsigned o = __shfl_xor_sync(0xffffffffu, m, off);
                m = o > m ? o : m;
            }
        }
        const bool mine = best == m;
        const unsigned who = (__ballot_sync(0xffffffffu, mine) >> lane0) & kMask;
        const bool ambiguous = (who & (who - 1u)) != 0u || (mine && tie);
        if (__any_sync(0xffffffffu, ambiguous)) {
            p = smem_pivot_exact<T>(M, RS, k, lo, hi, t, lim);
            cv = TL_SM(M, p * RS + k, lim);
            __syncwarp();  // before the interchange writes the column
        } else {
            const int w = lane0 + __ffs(static_cast<int>(who)) - 1;
            p = __shfl_sync(0xffffffffu, row, w);
            cv = __shfl_sync(0xffffffffu, v, w);
        }
    }
};

// Rows (multipliers) of one lane per pass: every row of its share in one
// pass from 8 lanes on.
template <int T>
struct RowChunk {
    static constexpr int U = TL_MAX_N / T < 4 ? TL_MAX_N / T : 4;
};

// Candidates of column k in rows [lo, hi) from shared memory.
template <int T>
__device__ __forceinline__ void smem_scan(const double *M, int RS, int k, int lo, int hi, int t, int lim, PivotScan &sc)
{
    constexpr int U = RowChunk<T>::U;
    sc.clear();
#pragma unroll 1
    for (int ib = lo; ib < hi; ib += U * T) {
        double v[U];
#pragma unroll
        for (int c = 0; c < U; ++c) {
            const int i = ib + t + c * T;
            v[c] = i < hi ? TL_SM(M, i * RS + k, lim) : 0.0;
        }
#pragma unroll
        for (int c = 0; c < U; ++c) sc.add(v[c], ib + t + c * T, ib + t + c * T < hi);
        if (U * T >= TL_MAX_N) break;
    }
}

// Rows the pivot of step k is sought in first (the whole column, or with
// tile-local pivoting the diagonal tile).
__device__ __forceinline__ int smem_pivot_limit(int n, int k, int tile)
{
    return tile > 0 && tile < n ? min(n, (k / tile + 1) * tile) : n;
}

// The pivot of step k from the group's candidates in rows [k, hi); with
// tile-local pivoting a best magnitude below the threshold (in some group
// of the warp) takes the first maximum over the whole column instead.
template <int T>
__device__ __forceinline__ void smem_pivot(const double *M, int n, int RS, int k, int hi, int t, int lim,
                                           double threshold, const PivotScan &sc, int *piv, double &cv, int &p, int &info)
{
    sc.finish<T>(M, RS, k, k, hi, t, lim, cv, p);
    if (hi < n && __any_sync(0xffffffffu, dev::mag_bits(cv) < dev::mag_bits(threshold))) {
        const int p2 = smem_pivot_exact<T>(M, RS, k, k, n, t, lim);
        if (dev::mag_bits(cv) < dev::mag_bits(threshold)) {
            p = p2;
            cv = TL_SM(M, p2 * RS + k, lim);
        }
        __syncwarp();
    }
    if (dev::mag_bits(cv) == 0ULL && info == 0) info = k + 1;
    if (t == 0) TL_SM(piv, k, n) = p;
}

// Interchange rows k and p over the columns [jlo, wcols), the entries of a
// pass loaded before its first store.  PEND (the second step of a pair, row
// k = kp + 1): columns from kp + 2 on of the row that becomes row k receive
// step kp on the way (l: its negated multiplier, upd: unless step kp's pivot
// was zero).  worst collects the largest high word of |.| of the new row k.
template <int T, bool PEND>
__device__ __forceinline__ void smem_swap(double *M, int n, int RS, int k, int p, int t, int lim, int jlo, int wcols,
                                          double l, bool upd, unsigned &worst)
{
    constexpr int U = T == 32 ? 2 : T == 16 ? 3 : T == 8 ? 5 : 4;
    const int first = PEND ? k + 1 : jlo;
    const int rk = k * RS, rp = p * RS, ru = (k - 1) * RS;
    if (PEND) {  // the columns without an update
        for (int j = jlo + t; j < first; j += T) {
            const double vk = TL_SM(M, rk + j, lim);
            TL_SM(M, rk + j, lim) = TL_SM(M, rp + j, lim);
            TL_SM(M, rp + j, lim) = vk;
        }
    }
#pragma unroll 1
    for (int jb = first; jb < wcols; jb += U * T) {
        double vk[U], vp[U], u[U];
#pragma unroll
        for (int c = 0; c < U; ++c) {
            const int j = jb + t + c * T;
            const bool in = j < wcols;
            vk[c] = in ? TL_SM(M, rk + j, lim) : 0.0;
            vp[c] = in ? TL_SM(M, rp + j, lim) : 0.0;
            if (PEND) u[c] = in ? TL_SM(M, ru + j, lim) : 0.0;
        }
#pragma unroll
        for (int c = 0; c < U; ++c) {
            // a branch the whole warp takes: an FP64 instruction of which no
            // lane is active still takes the pipe for its 64 clocks
            if (jb + c * T >= wcols) break;
            const int j = jb + t + c * T;
            const unsigned hi = static_cast<unsigned>(dev::mag_bits(vp[c]) >> 32);
            worst = (j < n && hi > worst) ? hi : worst;
            if (PEND) vp[c] = dev::sel(upd, __fma_rn(l, u[c], vp[c]), vp[c]);
            if (j < wcols) {
                TL_SM(M, rp + j, lim) = vk[c];
                TL_SM(M, rk + j, lim) = vp[c];
            }
        }
        if (U * T > TL_MAX_N) break;
    }
}

// Multiplier of a step whose pivot is zero (a sign flip) or below DBL_MIN
// (a quotient) in some group of the warp; out of line.
static __device__ __noinline__ double smem_rare_multiplier(double a, double cv, double nr, bool zero, bool small)
{
    return zero ? dev::neg(a) : small ? __ddiv_rn(a, dev::neg(cv)) : __dmul_rn(a, nr);
}

// Negated multipliers of column k below row k; with UPD the same lane also
// applies step k to the entry of column k + 1 of its row and proposes it as a
// pivot candidate of step k + 1 (rows below hi).
template <int T, bool UPD>
__device__ __forceinline__ void smem_multipliers(double *M, int n, int RS, int k, int t, int lim, double cv, double nr,
                                                 bool zero, bool small, int hi, PivotScan &sc)
{
    constexpr int U = RowChunk<T>::U;
    const double ukk1 = UPD ? TL_SM(M, k * RS + k + 1, lim) : 0.0;
    const bool rare = __any_sync(0xffffffffu, small || zero);
    if (UPD) sc.clear();
#pragma unroll 1
    for (int ib = k + 1; ib < n; ib += U * T) {
        double a[U], b[U];
#pragma unroll
        for (int c = 0; c < U; ++c) {
            const int i = ib + t + c * T;
            a[c] = i < n ? TL_SM(M, i * RS + k, lim) : 0.0;
            if (UPD) b[c] = i < n ? TL_SM(M, i * RS + k + 1, lim) : 0.0;
        }
#pragma unroll
        for (int c = 0; c < U; ++c) {
            if (ib + c * T >= n) break;  // the same on every lane
            const int i = ib + t + c * T;
            const double l = rare ? smem_rare_multiplier(a[c], cv, nr, zero, small) : __dmul_rn(a[c], nr);
            if (i < n) TL_SM(M, i * RS + k, lim) = l;
            if (UPD) {
                const double w = dev::sel(zero, b[c], __fma_rn(l, ukk1, b[c]));
                if (i < n) TL_SM(M, i * RS + k + 1, lim) = w;
                sc.add(w, i, i < hi);
            }
        }
        if (U * T >= TL_MAX_N) break;
    }
}

// Returns info; worst receives the largest high word of the magnitudes of
// A's entries and of the values that replaced them, as this lane met them: a
// non-finite entry of A stays non-finite until it is the pivot or in a row of
// U, or, below a smaller pivot that is not zero, until its multiplier has
// spread along its row.  A zero pivot above such an entry, which tile-local
// pivoting with a threshold of 0 keeps, spreads it nowhere: a system with a
// zero pivot reports 0x7ff00000 there.  So only when some lane of the group
// reports 0x7ff00000 or more can A hold a non-finite entry.
template <int T, bool SOLVE, bool KEEPL>
__device__ __forceinline__ int smem_lupp2(double *M, int n, int RS, int t, int tile, double threshold, unsigned &worst)
{
    static_assert(T >= 1 && T <= 32 && (32 % T) == 0, "T must divide 32");
    const int lane0 = (static_cast<int>(threadIdx.x) & 31) - t;
    const int lim = smem_piv_offset(n) + (n + 1) / 2;  // doubles in the system's block
    double *rcp = M + n * RS;                           // n doubles
    int *piv = reinterpret_cast<int *>(rcp + n);        // n ints
    int info = 0;
    bool tiny = false;
    worst = 0;
    const int wcols = n + (SOLVE ? 1 : 0);              // columns incl. b
    auto note = [&](double v) {
        const unsigned hi = static_cast<unsigned>(dev::mag_bits(v) >> 32);
        worst = hi > worst ? hi : worst;
    };
    PivotScan sc;
    int k = 0;
    for (; k + 1 < n; k += 2) {
        // ---- step k: pivot, reciprocal and interchange, multipliers, column
        //      k+1 with the candidates of step k+1 ----
        const int hi0 = smem_pivot_limit(n, k, tile);
        smem_scan<T>(M, RS, k, k, hi0, t, lim, sc);
        double cv;
        int p;
        smem_pivot<T>(M, n, RS, k, hi0, t, lim, threshold, sc, piv, cv, p, info);
        note(cv);
        const bool z0 = dev::mag_bits(cv) == 0ULL;
        const bool s0 = !z0 && dev::mag_bits(cv) < dev::kDblMinBits;
        smem_swap<T, false>(M, n, RS, k, p, t, lim, KEEPL ? 0 : k, wcols, 0.0, false, worst);
        const double r0 = dev::rcp_rn(cv);
        if (t == 0) TL_SM(rcp, k, n) = r0;
        tiny = tiny || s0;
        __syncwarp();
        const int k1 = k + 1;
        const int hi1 = smem_pivot_limit(n, k1, tile);
        smem_multipliers<T, true>(M, n, RS, k, t, lim, cv, dev::neg(r0), z0, s0, hi1, sc);
        __syncwarp();
        // ---- step k+1: pivot, interchange of rows that still carry step k's
        //      pending update and -l_ik (the new row k+1 receives it on the
        //      way), multipliers ----
        double cv1;
        int p1;
        smem_pivot<T>(M, n, RS, k1, hi1, t, lim, threshold, sc, piv, cv1, p1, info);
        note(cv1);
        const bool z1 = dev::mag_bits(cv1) == 0ULL;
        const bool s1 = !z1 && dev::mag_bits(cv1) < dev::kDblMinBits;
        const double lp = TL_SM(M, p1 * RS + k, lim);
        __syncwarp();
        smem_swap<T, true>(M, n, RS, k1, p1, t, lim, KEEPL ? 0 : k, wcols, lp, !z0, worst);
        const double r1 = dev::rcp_rn(cv1);
        if (t == 0) TL_SM(rcp, k1, n) = r1;
        tiny = tiny || s1;
        __syncwarp();
        smem_multipliers<T, false>(M, n, RS, k1, t, lim, cv1, dev::neg(r1), z1, s1, n, sc);
        __syncwarp();
        // ---- both updates of the block rows k+2.., columns k+2.. ----
        const int ncols = wcols - (k + 2);
        const int nrows = n - (k + 2);
        const int nel = nrows * ncols;
        if (nel > 0) {
            const int q = div_small(T, ncols), rq = T - q * ncols;   // (row, column) advance per stride
            int ei = div_small(t, ncols);
            int ej = t - ei * ncols;                                 // element t: row k+2+ei, column k+2+ej
            const int u0 = k * RS + k + 2;                          // rows k and k+1 from column k+2
            const int u1 = k1 * RS + k + 2;
            if (!__any_sync(0xffffffffu, z0 || z1)) {
                for (int e = t; e < nel; e += T) {
                    const int ri = (k + 2 + ei) * RS;
                    double a = TL_SM(M, ri + k + 2 + ej, lim);
                    a = __fma_rn(TL_SM(M, ri + k, lim), TL_SM(M, u0 + ej, lim), a);
                    a = __fma_rn(TL_SM(M, ri + k1, lim), TL_SM(M, u1 + ej, lim), a);
                    TL_SM(M, ri + k + 2 + ej, lim) = a;
                    ej += rq;
                    ei += q;
                    if (ej >= ncols) {
                        ej -= ncols;
                        ++ei;
                    }
                }
            } else {  // a zero pivot in some group: that step leaves the block as it is
                for (int e = t; e < nel; e += T) {
                    const int ri = (k + 2 + ei) * RS;
                    double a = TL_SM(M, ri + k + 2 + ej, lim);
                    if (!z0) a = __fma_rn(TL_SM(M, ri + k, lim), TL_SM(M, u0 + ej, lim), a);
                    if (!z1) a = __fma_rn(TL_SM(M, ri + k1, lim), TL_SM(M, u1 + ej, lim), a);
                    TL_SM(M, ri + k + 2 + ej, lim) = a;
                    ej += rq;
                    ei += q;
                    if (ej >= ncols) {
                        ej -= ncols;
                        ++ei;
                    }
                }
            }
        }
        __syncwarp();
    }
    if (k < n) {  // odd n: the last step (one row: its own pivot)
        const double cv = TL_SM(M, k * RS + k, lim);
        note(cv);
        if (dev::mag_bits(cv) == 0ULL && info == 0) info = k + 1;
        const bool s0 = dev::mag_bits(cv) != 0ULL && dev::mag_bits(cv) < dev::kDblMinBits;
        const double r0 = dev::rcp_rn(cv);
        if (t == 0) {
            TL_SM(piv, k, n) = k;
            TL_SM(rcp, k, n) = r0;
        }
        tiny = tiny || s0;
        __syncwarp();
    }

    if (tile > 0 && info != 0) worst = 0x7ff00000u;

    // a6 (back part): x_i = y_i * RN(1/u_ii) (y_i / u_ii when a pivot was
    // below DBL_MIN), then y_r -= u_ri x_i for r < i
    if (SOLVE) {
        const bool any_tiny = __any_sync(0xffffffffu, tiny);
        if constexpr (T >= 4) {
            // y in registers (lane t holds rows t, t + T, ...); the next
            // column of U and the next reciprocal are loaded before the
            // product of the current row
            constexpr int KM = TL_MAX_N / T;  // row slots per lane
            double y[KM], u[KM];
#pragma unroll
            for (int s = 0; s < KM; ++s) {
                const int r = t + s * T;
                y[s] = r < n ? TL_SM(M, r * RS + n, lim) : 0.0;
                u[s] = r < n - 1 ? TL_SM(M, r * RS + n - 1, lim) : 0.0;
            }
            double rc = TL_SM(rcp, n - 1, n);
#pragma unroll 1
            for (int i = n - 1; i >= 0; --i) {
                const int owner = i % T, slot = i / T;
                double yi = y[0];
#pragma unroll
                for (int s = 1; s < KM; ++s) yi = dev::sel(s == slot, y[s], yi);
                double xi;
                if (!any_tiny) xi = __dmul_rn(yi, rc);
                else xi = tiny ? __ddiv_rn(yi, TL_SM(M, i * RS + i, lim)) : __dmul_rn(yi, rc);
                double un[KM];
#pragma unroll
                for (int s = 0; s < KM; ++s) {
                    const int r = t + s * T;
                    un[s] = r < i - 1 ? TL_SM(M, r * RS + i - 1, lim) : 0.0;
                }
                rc = TL_SM(rcp, i > 0 ? i - 1 : 0, n);
                xi = __shfl_sync(0xffffffffu, xi, lane0 + owner);
#pragma unroll
                for (int s = 0; s < KM; ++s) y[s] = dev::sel(t == owner && s == slot, xi, y[s]);
                const double nxi = dev::neg(xi);
#pragma unroll
                for (int s = 0; s < KM; ++s) {
                    if (s * T >= i) break;  // no row of this slot lies above row i
                    if (t + s * T < i) y[s] = __fma_rn(u[s], nxi, y[s]);
                }
#pragma unroll
                for (int s = 0; s < KM; ++s) u[s] = un[s];
            }
#pragma unroll
            for (int s = 0; s < KM; ++s) {
                const int r = t + s * T;
                if (r < n) TL_SM(M, r * RS + n, lim) = y[s];
            }
            __syncwarp();
        } else {
            for (int i = n - 1; i >= 0; --i) {
                if (t == 0) {
                    const double y = TL_SM(M, i * RS + n, lim);
                    double xi;
                    if (!any_tiny) xi = __dmul_rn(y, TL_SM(rcp, i, n));
                    else xi = tiny ? __ddiv_rn(y, TL_SM(M, i * RS + i, lim)) : __dmul_rn(y, TL_SM(rcp, i, n));
                    TL_SM(M, i * RS + n, lim) = xi;
                }
                __syncwarp();
                const double nxi = dev::neg(TL_SM(M, i * RS + n, lim));
                for (int r2 = t; r2 < i; r2 += T)
                    TL_SM(M, r2 * RS + n, lim) = __fma_rn(TL_SM(M, r2 * RS + i, lim), nxi, TL_SM(M, r2 * RS + n, lim));
                __syncwarp();
            }
        }
    }
    return info;
}

// Whether some entry of a group's system (nn consecutive doubles at A, null
// without a system) is not finite, read only when some group of the warp
// suspects it (see smem_lupp2).
template <int T>
__device__ __forceinline__ bool smem_bad_input(bool suspect, const double *A, int nn, int t)
{
    if (!__any_sync(0xffffffffu, suspect)) return false;
    int badv = 0;
    if (A)
        for (int e = t; e < nn; e += T) badv |= dev::is_nonfinite(A[e]) ? 1 : 0;
    return group_any_int<T>(badv) != 0;
}

// MODE: kGesv (A const, b -> x, LU optional by KEEP) or kGetrf (A in place).
// WALK: element walk of the trailing update instead of the lane tile.
template <int T, int LAYOUT, int MODE, bool KEEP, bool WALK = (T >= 16)>
__global__ void __launch_bounds__(128) k_smem_group(SolveArgs args, int n)
{
    extern __shared__ double smem[];
    const int SB = blockDim.x / T;                 // systems per block
    const int per = smem_sys_doubles(n, T);
    const int RS = smem_row_stride(n);            // row stride
    const int64_t s0 = static_cast<int64_t>(blockIdx.x) * SB;
    const double *Ag = (MODE == kGetrf) ? args.LU : args.A;
    const int nn = n * n;
    const unsigned m20 = magic20(n);

    // ---- load, all copies in flight at once (cp.async).  Interleaved: thread
    //      (q = tid % SB, tp = tid / SB) copies entries tp, tp+T, ... of
    //      system s0+q (coalesced over q); per system: a warp copies 32
    //      consecutive entries of one system at a time ----
    if (LAYOUT == kInterleaved) {
        const int q = threadIdx.x % SB;
        const int tp = threadIdx.x / SB;
        const int64_t s = s0 + q;
        double *M = smem + q * per;
        if (s < args.batch) {
            for (int e = tp; e < nn; e += T) {
                const int j = div20(e, m20);
                cp_async8(&TL_SM(M, (e - j * n) * RS + j, per), Ag + static_cast<int64_t>(e) * args.ld + s);
            }
            if (MODE == kGesv)
                for (int i2 = tp; i2 < n; i2 += T)
                    cp_async8(&TL_SM(M, i2 * RS + n, per), args.b + static_cast<int64_t>(i2) * args.ld + s);
        }
    } else {
        const int lane = threadIdx.x & 31;
        for (int q = threadIdx.x >> 5; q < SB && s0 + q < args.batch; q += blockDim.x >> 5) {
            double *M = smem + q * per;
            const double *src = Ag + (s0 + q) * nn;
            for (int e = lane; e < nn; e += 32) {
                const int j = div20(e, m20);
                cp_async8(&TL_SM(M, (e - j * n) * RS + j, per), src + e);
            }
            if (MODE == kGesv && lane < n) cp_async8(&TL_SM(M, lane * RS + n, per), args.b + (s0 + q) * n + lane);
        }
    }
    // the systems of the block one wave of resident blocks ahead, which takes
    // a slot of shared memory when this one gives it up, into L2 (n = 19
    // interleaved, 150,001 systems: 901 -> 891 us)
    if (static_cast<int64_t>(blockIdx.x) + args.ahead < gridDim.x) {
        const int64_t sn = s0 + args.ahead * SB;
        const int64_t last = args.batch - sn < SB ? args.batch - sn : SB;  // systems
        if (LAYOUT == kInterleaved) {
            for (int e = threadIdx.x; e < nn; e += blockDim.x) prefetch_l2(Ag + static_cast<int64_t>(e) * args.ld + sn);
        } else {
            for (int64_t e = threadIdx.x * 16; e < last * nn; e += blockDim.x * 16) prefetch_l2(Ag + sn * nn + e);
        }
    }
    cp_async_wait_all();
    __syncthreads();

    // ---- compute: lanes t = lane % T of a group own system q ----
    const int lane = threadIdx.x & 31;
    const int t = lane % T;
    const int q = threadIdx.x / T;
    const int64_t s = s0 + q;
    const bool active = s < args.batch;
    double *M = smem + q * per;
    const int *piv = reinterpret_cast<const int *>(M + smem_piv_offset(n));  // pivots (after n reciprocals)
    bool bad = false;
    int info;
    if constexpr (WALK) {
        unsigned worst = 0;
        info = smem_lupp2<T, MODE == kGesv, KEEP || MODE == kGetrf>(M, n, RS, t, args.tile, args.threshold, worst);
        // only a system that met a non-finite value can have one in A; whether
        // it has (or overflowed on the way) is read from A again
        const bool suspect = active && worst >= 0x7ff00000u;
        if (__any_sync(0xffffffffu, suspect)) {
            int badv = 0;
            if (active) {
                const double *src = Ag + (LAYOUT == kInterleaved ? s : s * nn);
                const int64_t es = LAYOUT == kInterleaved ? args.ld : 1;
                for (int e = t; e < nn; e += T) badv |= dev::is_nonfinite(src[e * es]) ? 1 : 0;
            }
            bad = group_any_int<T>(badv) != 0;
        }
    } else {
        int badv = 0;
        if (active) {
            for (int e = t; e < nn; e += T) {
                const int j = div20(e, m20);
                badv |= dev::is_nonfinite(M[(e - j * n) * RS + j]) ? 1 : 0;
            }
        }
        bad = group_any_int<T>(badv) != 0;
        info = smem_lupp<T, MODE == kGesv>(M, n, RS, t, args.tile, args.threshold);
    }
    if (bad) info = -1;

    // a7: store
    if (active) {
        for (int i = t; i < n; i += T) {
            const int64_t vi = (LAYOUT == kInterleaved) ? static_cast<int64_t>(i) * args.ld + s : s * n + i;
            if (MODE == kGesv) st_stream(args.x + vi, info != 0 ? dev::nan_value() : M[i * RS + n]);
            st_stream(args.ipiv + vi, bad ? i + 1 : piv[i] + 1);
        }
        if (t == 0) st_stream(args.info + s, info);
    }
    if constexpr (KEEP) {
        // the factors by the mapping of the loads (a group's own entries of
        // one column lie in as many rows of the interleaved storage: 50,000
        // systems of n = 13 145 us that way, 131 us now); the slot of the first
        // reciprocal tells the block whether the system had bad input
        if (t == 0) M[smem_rcp_offset(n)] = bad ? 1.0 : 0.0;
        __syncthreads();
        // entries e0, e0 + step, ... of system qs, entry e at LU[e * es + base]
        auto store = [&](int qs, int e0, int step, int64_t base, int64_t es) {
            const double *Mq = smem + qs * per;
            if (Mq[smem_rcp_offset(n)] == 0.0) {
#pragma unroll 4
                for (int e = e0; e < nn; e += step) {
                    const int j = div20(e, m20), i = e - j * n;
                    const double v = Mq[i * RS + j];
                    st_stream(args.LU + (base + e * es), j < i ? dev::neg(v) : v);
                }
            } else if (MODE == kGesv) {  // nothing is factored: A
                for (int e = e0; e < nn; e += step) args.LU[base + e * es] = args.A[base + e * es];
            }
        };
        if (LAYOUT == kInterleaved) {
            const int qs = threadIdx.x % SB;
            if (s0 + qs < args.batch) store(qs, threadIdx.x / SB, T, s0 + qs, args.ld);
        } else {
            for (int qs = threadIdx.x >> 5; qs < SB && s0 + qs < args.batch; qs += blockDim.x >> 5)
                store(qs, lane, 32, (s0 + qs) * nn, 1);
        }
    }
}

// Ragged batches (tl_lupp_solve_batched): persistent over the bucket of
// systems of size n (run-time), SB = blockDim/T systems per block and trip;
// each system at its own offsets in per-system column-major storage.
// Binary64, element walk (smem_lupp2).
template <int T>
__global__ void __launch_bounds__(128) k_smem_ragged(RaggedArgs r, int n)
{
    extern __shared__ double smem[];
    const int SB = blockDim.x / T;
    const int per = smem_sys_doubles(n, T);
    const int RS = smem_row_stride(n);
    const int nn = n * n;
    const unsigned m20 = magic20(n);
    const int64_t beg = r.offsets[n];
    const int64_t full = r.offsets[n + 1] - beg;
    int64_t count = full;
    if (r.counts) {
        const int64_t c = r.counts[n];
        count = c < 0 ? 0 : (c < full ? c : full);
    }
    const int lane = threadIdx.x & 31;
    const int t = lane % T;
    const int q = threadIdx.x / T;
    for (int64_t base = static_cast<int64_t>(blockIdx.x) * SB; base < count;
         base += static_cast<int64_t>(gridDim.x) * SB) {           // block-uniform trip
        // load: thread (qL = tid % SB, tp = tid / SB) copies elements
        // e = tp, tp+T, ... of system base+qL (cp.async)
        {
            const int qL = threadIdx.x % SB;
            const int tp = threadIdx.x / SB;
            double *M = smem + qL * per;
            if (base + qL < count) {
                const int64_t sidx = r.bucket[beg + base + qL];
                const double *A = r.A + r.a_off[sidx];
                for (int e = tp; e < nn; e += T) {
                    const int j = div20(e, m20);
                    cp_async8(&TL_SM(M, (e - j * n) * RS + j, per), A + e);
                }
                const double *bv = r.b + r.b_off[sidx];
                for (int i2 = tp; i2 < n; i2 += T) cp_async8(&TL_SM(M, i2 * RS + n, per), bv + i2);
            }
            cp_async_wait_all();
        }
        __syncthreads();
        const bool active = base + q < count;
        double *M = smem + q * per;
        unsigned worst = 0;
        int info = smem_lupp2<T, true, false>(M, n, RS, t, 0, 0.0, worst);
        const bool bad = smem_bad_input<T>(active && worst >= 0x7ff00000u,
                                           active ? r.A + r.a_off[r.bucket[beg + base + q]] : nullptr, nn, t);
        if (bad) info = -1;
        if (active) {
            const int64_t sidx = r.bucket[beg + base + q];
            const int *piv = reinterpret_cast<const int *>(M + smem_piv_offset(n));
            double *x = r.x + r.b_off[sidx];
            int32_t *ip = r.ipiv + r.piv_off[sidx];
            for (int i = t; i < n; i += T) {
                st_stream(x + i, info != 0 ? dev::nan_value() : M[i * RS + n]);
                st_stream(ip + i, bad ? i + 1 : piv[i] + 1);
            }
            if (t == 0) st_stream(r.info + sidx, info);
        }
        __syncthreads();  // the next trip's loads overwrite the blocks
    }
}

}  // namespace tl
