// tl_getrs.cuh -- solves with given factors, the factors in shared memory,
// run-time n: y = P b, L y' = y, U x = y' (Sec. 2.2, the getrs part).
//
// The FP64 pipe takes 64 clocks of a sub-partition per warp instruction
// whatever the number of active lanes, so lanes are what counts:
//   * k_getrs_rhs: one thread per right-hand side.  Every lane runs its own
//     substitution (n^2 instructions, all lanes useful); the right-hand sides
//     of a block's systems are dealt to its threads without gaps.
//   * k_getrs_rows<T>: for one or two right-hand sides, where a thread each
//     would leave shared memory room for one warp: T lanes per system, lane t
//     holding rows t, t + T, ... of y in registers.
// Both copy the factors once (cp.async), form the reciprocals RN(1/u_ii) and
// the row order of P together, and apply the updates of every entry in the
// order of the register kernels: forward in increasing, back in decreasing
// column order.
#pragma once
#include "tinylu.h"
#include "tl_bounds.cuh"
#include "tl_getrs_plan.h"
#include "tl_kernels.cuh"
#include "tl_smem.cuh"

namespace tl {

// Copy the factors of `live` systems from s0 on into shared memory
// (system q at q * per) and form their reciprocals and row orders.  All
// threads of the block; flags[q] becomes 1 when a pivot is below DBL_MIN.
template <int LAYOUT>
__device__ __forceinline__ void getrs_load(const SolveArgs &args, int n, int64_t s0, int live, int SB, double *smem,
                                           int per, int *flags)
{
    const int RS = getrs_row_stride(n), nn = n * n;
    const unsigned m20 = magic20(n);
    const int tid = static_cast<int>(threadIdx.x), nth = static_cast<int>(blockDim.x);
    for (int q = tid; q < SB; q += nth) flags[q] = 0;
    if (LAYOUT == kInterleaved) {
        // consecutive threads copy the same entry of consecutive systems
        const int width = SB < nth ? SB : nth, rows = nth / width;
        const int q0 = tid % width, e0 = tid / width;
        if (e0 < rows)
            for (int q = q0; q < live; q += width)
                for (int e = e0; e < nn; e += rows) {
                    const int j = div20(e, m20);
                    cp_async8(&TL_SM(smem, q * per + (e - j * n) * RS + j, SB * per),
                              args.A + static_cast<int64_t>(e) * args.ld + s0 + q);
                }
    } else {
        const int warp = tid >> 5, nw = nth >> 5, lane = tid & 31;
        for (int q = warp; q < live; q += nw) {
            const double *src = args.A + (s0 + q) * nn;
            for (int e = lane; e < nn; e += 32) {
                const int j = div20(e, m20);
                cp_async8(&TL_SM(smem, q * per + (e - j * n) * RS + j, SB * per), src + e);
            }
        }
    }
    // pivots behind the reciprocals while the copies are in flight
    for (int e = tid; e < live * n; e += nth) {
        const int q = LAYOUT == kInterleaved ? e % live : e / n, k = LAYOUT == kInterleaved ? e / live : e % n;
        int *row = reinterpret_cast<int *>(smem + q * per + n * RS + n);
        const int p =
            args.ipiv[LAYOUT == kInterleaved ? static_cast<int64_t>(k) * args.ld + s0 + q : (s0 + q) * n + k] - 1;
        row[k] = p > k && p < n ? p : k;  // what getrf never writes is no interchange (row indexes memory)
    }
    cp_async_wait_all();
    __syncthreads();
    // reciprocals; source row of every row of P b: the interchanges k = 0, 1,
    // ... traced backwards
    for (int eb = 0; eb < live * n; eb += nth) {
        const int e = eb + tid, q = e / n, i = e - q * n;
        const bool in = e < live * n;
        double u = 1.0;
        if (in) u = TL_SM(smem, q * per + i * RS + i, SB * per);
        const double r = dev::rcp_rn(u);
        if (in) {
            TL_SM(smem, q * per + n * RS + i, SB * per) = r;
            if (dev::mag_bits(u) < dev::kDblMinBits) flags[q] = 1;
        }
    }
    for (int e = tid; e < live * n; e += nth) {
        const int q = e / n, i = e - q * n;
        int *piv = reinterpret_cast<int *>(smem + q * per + n * RS + n);
        int src = i;
        for (int k = n - 1; k >= 0; --k) {
            const int p = piv[k];
            src = src == k ? p : (src == p ? k : src);
        }
        piv[n + i] = src;
    }
    __syncthreads();
}

// One thread per right-hand side: block of SB systems, thread tid solves
// one right-hand side (neighbours: consecutive systems interleaved,
// consecutive right-hand sides per system).  Behind the SB systems shared
// memory holds every thread's y, negated (entry i at i * threads + tid).
template <int LAYOUT>
__global__ void __launch_bounds__(128) k_getrs_rhs(SolveArgs args, int n, int SB)
{
    extern __shared__ double smem[];
    const int per = getrs_sys_doubles(n), RS = getrs_row_stride(n);
    const int tid = static_cast<int>(threadIdx.x), nth = static_cast<int>(blockDim.x);
    int *flags = reinterpret_cast<int *>(smem + SB * per);
    double *Y = smem + getrs_block_doubles(n, SB) + tid;
    const int64_t s0 = static_cast<int64_t>(blockIdx.x) * SB;
    const int live = static_cast<int>(args.batch - s0 < SB ? args.batch - s0 : SB);
    getrs_load<LAYOUT>(args, n, s0, live, SB, smem, per, flags);
    const int q = LAYOUT == kInterleaved ? tid % SB : tid / args.nrhs;
    const int r = LAYOUT == kInterleaved ? tid / SB : tid - q * args.nrhs;
    if (q >= live || r >= args.nrhs) return;
    const int ylim = (n - 1) * nth + 1;  // doubles from Y[0] to this thread's last entry
    const double *M = smem + q * per;
    const double *rcp = M + n * RS;
    const int *row = reinterpret_cast<const int *>(rcp + n) + n;
    const int64_t s = s0 + q;
    const int64_t es = LAYOUT == kInterleaved ? args.ld : 1;
    double *B = args.x + (LAYOUT == kInterleaved ? static_cast<int64_t>(r) * n * args.ld + s
                                                 : (s * args.nrhs + r) * static_cast<int64_t>(n));
    // forward: y_i = b_row(i) - sum_{j < i} l_ij y_j
    for (int i = 0; i < n; ++i) {
        double v = B[TL_SM(row, i, n) * es];
        const int ri = i * RS;
#pragma unroll 4
        for (int j = 0; j < i; ++j) v = __fma_rn(TL_SM(M, ri + j, per), TL_SM(Y, j * nth, ylim), v);
        TL_SM(Y, i * nth, ylim) = dev::neg(v);
    }
    // back: x_i = (y_i - sum_{j > i} u_ij x_j) * RN(1/u_ii), a quotient when a
    // pivot of the system is below DBL_MIN
    const bool tiny = flags[q] != 0;
    for (int i = n - 1; i >= 0; --i) {
        double v = dev::neg(TL_SM(Y, i * nth, ylim));
        const int ri = i * RS;
#pragma unroll 4
        for (int j = n - 1; j > i; --j) v = __fma_rn(TL_SM(M, ri + j, per), TL_SM(Y, j * nth, ylim), v);
        v = tiny ? __ddiv_rn(v, TL_SM(M, ri + i, per)) : __dmul_rn(v, TL_SM(rcp, i, n));
        TL_SM(Y, i * nth, ylim) = dev::neg(v);
        B[i * es] = v;
    }
}

// T lanes per system with KM row slots each ((KM - 1) T < n <= KM T), nrhs
// right-hand sides one after another, interleaved storage.
template <int T, int KM>
__global__ void __launch_bounds__(128) k_getrs_rows(SolveArgs args, int n, int)
{
    extern __shared__ double smem[];
    const int SB = static_cast<int>(blockDim.x) / T;
    const int per = getrs_sys_doubles(n), RS = getrs_row_stride(n);
    int *flags = reinterpret_cast<int *>(smem + SB * per);
    const int64_t s0 = static_cast<int64_t>(blockIdx.x) * SB;
    const int live = static_cast<int>(args.batch - s0 < SB ? args.batch - s0 : SB);
    getrs_load<kInterleaved>(args, n, s0, live, SB, smem, per, flags);
    const int lane = threadIdx.x & 31, t = lane % T, lane0 = lane - t;
    const int q = static_cast<int>(threadIdx.x) / T;
    const bool active = q < live;
    const int64_t s = s0 + q;
    const double *M = smem + (active ? q : 0) * per;
    const double *rcp = M + n * RS;
    const int *row = reinterpret_cast<const int *>(rcp + n) + n;
    const bool tiny = active && flags[q] != 0;
    const bool any_tiny = __any_sync(0xffffffffu, tiny);
    const int64_t es = args.ld;
    for (int r = 0; r < args.nrhs; ++r) {
        double *B = args.x + static_cast<int64_t>(r) * n * args.ld + s;
        double y[KM], l[KM];
#pragma unroll
        for (int c = 0; c < KM; ++c) {
            const int i = t + c * T;
            y[c] = active && i < n ? B[TL_SM(row, i, n) * es] : 0.0;
            l[c] = i < n ? TL_SM(M, i * RS, per) : 0.0;
        }
        // forward, column by column (the next column loaded ahead)
#pragma unroll 1
        for (int k = 0; k + 1 < n; ++k) {
            const int owner = k % T, slot = k / T;
            double yk = y[0];
#pragma unroll
            for (int c = 1; c < KM; ++c) yk = dev::sel(c == slot, y[c], yk);
            const double nyk = dev::neg(__shfl_sync(0xffffffffu, yk, lane0 + owner));
            double ln[KM];
#pragma unroll
            for (int c = 0; c < KM; ++c) {
                const int i = t + c * T;
                ln[c] = i < n ? TL_SM(M, i * RS + k + 1, per) : 0.0;
            }
#pragma unroll
            for (int c = KM - 1; c >= 0; --c) {
                if (c * T + T - 1 <= k) break;  // no row of this slot lies below row k
                const int i = t + c * T;
                if (i > k && i < n) y[c] = __fma_rn(l[c], nyk, y[c]);
            }
#pragma unroll
            for (int c = 0; c < KM; ++c) l[c] = ln[c];
        }
        // back, column by column (l holds column n - 1)
        double rc = TL_SM(rcp, n - 1, n);
#pragma unroll 1
        for (int i = n - 1; i >= 0; --i) {
            const int owner = i % T, slot = i / T;
            double yi = y[0];
#pragma unroll
            for (int c = 1; c < KM; ++c) yi = dev::sel(c == slot, y[c], yi);
            double xi;
            if (!any_tiny) xi = __dmul_rn(yi, rc);
            else xi = tiny ? __ddiv_rn(yi, TL_SM(M, i * RS + i, per)) : __dmul_rn(yi, rc);
            double un[KM];
#pragma unroll
            for (int c = 0; c < KM; ++c) {
                const int j = t + c * T;
                un[c] = j < i - 1 ? TL_SM(M, j * RS + i - 1, per) : 0.0;
            }
            rc = TL_SM(rcp, i > 0 ? i - 1 : 0, n);
            xi = __shfl_sync(0xffffffffu, xi, lane0 + owner);
#pragma unroll
            for (int c = 0; c < KM; ++c) y[c] = dev::sel(t == owner && c == slot, xi, y[c]);
            const double nxi = dev::neg(xi);
#pragma unroll
            for (int c = 0; c < KM; ++c) {
                if (c * T >= i) break;  // no row of this slot lies above row i
                if (t + c * T < i) y[c] = __fma_rn(l[c], nxi, y[c]);
            }
#pragma unroll
            for (int c = 0; c < KM; ++c) l[c] = un[c];
        }
        __syncwarp();  // every lane has read its entries of b
        if (active) {
#pragma unroll
            for (int c = 0; c < KM; ++c) {
                const int i = t + c * T;
                if (i < n) B[i * es] = y[c];
            }
        }
    }
}

}  // namespace tl
