// tl_newton_smem.cu -- fused per-point Newton integration of the tanh law
// (Algorithm 2) for 11 <= n <= 32 with the Jacobian in shared memory: T
// lanes per point, 32 / T points per warp, the two-step element-walk LUpp
// of the shared-memory solver (smem_lupp2, run-time n).  Per iteration
// lane t of a point's group assembles rows t, t + T, ... of F and J
// (F_i = sum_j a_ij x_j + c_i tanh(x_i) - b_i with the sum as fma in
// increasing j; J = A + diag(c .* (1 - tanh^2 x))) into the augmented block
// [J | -F], the warp factors every group's block and solves for dx, and
// the group updates x.  Persistent: a group whose point stops stores it and
// takes the next one of its stride.
#include <cmath>

#include "tinylu.h"
#include "tl_handle.h"
#include "tl_internal.h"
#include "tl_newton.cuh"
#include "tl_smem.cuh"

namespace tl {
namespace {

// Warps per block: within 3% of 1 and 4 (measured at n = 10..32), and no
// size is left without room for a block.
constexpr int kWarpsPerBlock = 2;

// Lanes per point of the shared-memory kernel for the tanh law at size n;
// 0 where the sub-warp register kernel runs (n = 10; n <= 9 runs one
// thread per point).  Measured on GB300 (million points/s, 131,072 or 65,536
// points): n = 13: 4 lanes 65.3, 8 lanes 62.3; n = 18: 41.6, 42.7; n = 23:
// 8 lanes 25.0, 16 lanes 22.1; n = 25: 18.6, 18.4; n = 29: 11.5, 13.2; 32 lanes
// never for so many (n = 32: 9.8 against 10.6 with 16).  While there are few
// points a wider group shortens each of their steps, as in the fixed-size
// solves; a point's results are the same with any lane count.
int newton_smem_lanes(const tl_handle *h, int n, int64_t points)
{
    if (n <= 10 || n > TL_MAX_N) return 0;
    const int lanes = n <= 14 ? 4 : n <= 25 ? 8 : 16;
    for (int T : {32, 16, 8})
        if (T > lanes && points * T <= 32 * 16 * h->sm_count) return T;
    return lanes;
}

// Shared memory per point: the solver's block plus 32 doubles of x.
__host__ __device__ constexpr int newton_smem_doubles(int n, int T) { return smem_sys_doubles(n, T) + 32; }

// Whether |v| is infinite or NaN, on its high word.
__device__ __forceinline__ bool high_nonfinite(double v)
{
    return (static_cast<unsigned>(__double2hiint(v)) & 0x7ff00000u) == 0x7ff00000u;
}

// T lanes per point, 32 / T points per warp.  In every trip of the loop each
// group with a live point factors and solves its system [J | -F] (the warp
// together; groups without a point factor a stale block and ignore it),
// updates x, assembles the next system at the new x and decides; a group whose
// point stops stores it and takes the next one of its stride before the next
// trip, so no solve is idle while points are left.  At the first guess x = 0
// the system is A + diag(c) and -F = b: no products and no tanh are needed, so a
// new point costs copies (and the look for non-finite entries, whose products
// with 0 would be NaN).  A is copied into the block by cp.async, all entries in
// flight, while the lanes evaluate tanh; A x is then summed from there.
// Measured at n = 20 with 8 lanes, 65,537 points, against one assembly per
// trip with the entries loaded one by one and a trip without a solve at the end
// of each point: 2214 -> 1926 us.
template <int T>
__global__ void __launch_bounds__(32 * kWarpsPerBlock) k_newton_tanh_smem(NewtonBatch B, int n)
{
    extern __shared__ double smem[];
    constexpr int KM = TL_MAX_N / T;  // row slots per lane
    const int lane = threadIdx.x & 31;
    const int t = lane % T;
    const int per = newton_smem_doubles(n, T);
    double *M = smem + (threadIdx.x / T) * per;
    double *xs = M + smem_sys_doubles(n, T);
    const int RS = smem_row_stride(n);
    const int64_t ngroups = (static_cast<int64_t>(gridDim.x) * blockDim.x) / T;
    int64_t g = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) / T;
    bool have = g < B.total;
    const double *in = nullptr;
    int64_t np = 1, p = 0;
    double r0 = 0.0;
    int k = 0;

    // copy this lane's rows of A into the block
    auto copy_rows = [&]() {
        for (int i = t; i < n; i += T) {
            const double *src = in + static_cast<int64_t>(i) * np + p;
            const int64_t step = static_cast<int64_t>(n) * np;
            for (int j = 0; j < n; ++j, src += step) cp_async8(M + i * RS + j, src);
        }
    };
    // ||F||_2 from the squares of the lane's rows, by the same tree over 32
    // rows whatever T is (rows i and i + 16, then + 8, ...), so that a point's
    // decisions do not depend on the lanes that its launch gives it
    auto group_norm = [&](double (&sq)[KM]) {
#pragma unroll
        for (int off = 16; off >= T; off >>= 1)
#pragma unroll
            for (int s = 0; s < off / T; ++s) sq[s] += sq[s + off / T];
        double ss = sq[0];
#pragma unroll
        for (int off = T / 2; off >= 1; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
        return dev::sqrt_rn(ss);
    };
    auto store_point = [&](int st) {
        const NewtonJob jb = load_job(B, g);
        for (int i = t; i < n; i += T) jb.x[i * np + p] = xs[i];
        if (t == 0) {
            jb.iters[p] = k;
            jb.status[p] = st;
        }
        g += ngroups;
        have = g < B.total;
    };

    bool fresh = have;
    for (;;) {
        // groups without an assembled system take their next point, until it
        // needs a solve
        while (__any_sync(0xffffffffu, fresh)) {
            double sq[KM] = {};
            if (fresh) {
                const NewtonJob jb = load_job(B, g);
                in = jb.in;
                np = jb.npoints;
                p = g - jb.start;
                k = 0;
                copy_rows();
                cp_async_wait_all();
#pragma unroll
                for (int s = 0; s < KM; ++s) {
                    const int i = t + s * T;
                    if (i >= n) break;
                    xs[i] = 0.0;
                    const double ci = in[(n * n + i) * np + p];
                    const double bi = in[(n * n + n + i) * np + p];
                    bool bad = high_nonfinite(ci);
                    for (int j = 0; j < n; ++j) bad = bad || high_nonfinite(M[i * RS + j]);
                    M[i * RS + i] = __dadd_rn(M[i * RS + i], ci);
                    const double Fi = bad ? dev::nan_value() : 0.0 - bi;
                    M[i * RS + n] = dev::neg(Fi);
                    sq[s] = Fi * Fi;
                }
            }
            const double r = group_norm(sq);
            if (fresh) {
                r0 = r;
                const int st = newton_decide<32>(r, r0, 0, B.rtol, B.max_iter);
                if (st >= 0) store_point(st);
                fresh = st >= 0 && have;
            }
        }
        __syncwarp();
        if (!__any_sync(0xffffffffu, have)) break;
        // solve and update
        unsigned worst;  // a non-finite Jacobian shows in the next residual
        const int info = smem_lupp2<T, true, false>(M, n, RS, t, 0, 0.0, worst);
        int st = -1;
        if (have) {
            if (info != 0) {
                st = TL_NEWTON_SINGULAR;
            } else {
                for (int i = t; i < n; i += T) xs[i] += M[i * RS + n];
                ++k;
            }
        }
        __syncwarp();
        // the system at the new x
        const bool go = have && st < 0;
        double sq[KM] = {};
        if (go) copy_rows();
        double ti[KM];
#pragma unroll
        for (int s = 0; s < KM; ++s) {
            const int i = t + s * T;
            ti[s] = 0.0;
            if (go && i < n) ti[s] = tanh(xs[i]);
        }
        cp_async_wait_all();
#pragma unroll
        for (int s = 0; s < KM; ++s) {
            const int i = t + s * T;
            if (go && i < n) {
                const double ci = in[(n * n + i) * np + p];
                const double bi = in[(n * n + n + i) * np + p];
                double acc = 0.0;
#pragma unroll 4
                for (int j = 0; j < n; ++j) acc = fma(M[i * RS + j], xs[j], acc);
                M[i * RS + i] = fma(ci, fma(-ti[s], ti[s], 1.0), M[i * RS + i]);
                const double Fi = fma(ci, ti[s], acc) - bi;
                M[i * RS + n] = dev::neg(Fi);
                sq[s] = Fi * Fi;
            }
        }
        const double r = group_norm(sq);
        if (go) st = newton_decide<32>(r, r0, k, B.rtol, B.max_iter);
        __syncwarp();
        fresh = false;
        if (have && st >= 0) {
            store_point(st);
            fresh = have;
        }
    }
}

template <int T>
tl_status launch_smem_newton(tl_handle *h, int n, const NewtonBatch &B, cudaStream_t stream)
{
    const void *kern = reinterpret_cast<const void *>(&k_newton_tanh_smem<T>);
    int limit = 0;
    const tl_status st = smem_opt_in(h, kern, &limit);
    if (st != TL_OK) return st;
    const size_t smem = static_cast<size_t>(32 * kWarpsPerBlock / T) * newton_smem_doubles(n, T) * 8;
    if (smem > static_cast<size_t>(limit)) return TL_ERR_UNSUPPORTED;
    const int nb = blocks_per_sm(h, kern, 32 * kWarpsPerBlock, smem);
    const int64_t per_block = 32 * kWarpsPerBlock / T;
    const int64_t need = (B.total + per_block - 1) / per_block;
    const int64_t resident = static_cast<int64_t>(nb < 1 ? 1 : nb) * h->sm_count;
    const unsigned grid = static_cast<unsigned>(need < resident ? need : resident);
    NewtonBatch arg = B;
    int n_arg = n;
    void *params[] = {&arg, &n_arg};
    const cudaError_t e = cudaLaunchKernel(kern, dim3(grid), dim3(32 * kWarpsPerBlock), params, smem, stream);
    return e == cudaSuccess ? TL_OK : fail_cuda(h, e);
}

}  // namespace

// Shared-memory tanh Newton for the sizes newton_smem_lanes names (false
// for the others).
bool newton_tanh_smem_launch(tl_handle *h, int n, const NewtonBatch &B, cudaStream_t stream, tl_status *out)
{
    switch (newton_smem_lanes(h, n, B.total)) {
    case 4: *out = launch_smem_newton<4>(h, n, B, stream); return true;
    case 8: *out = launch_smem_newton<8>(h, n, B, stream); return true;
    case 16: *out = launch_smem_newton<16>(h, n, B, stream); return true;
    case 32: *out = launch_smem_newton<32>(h, n, B, stream); return true;
    default: return false;
    }
}

}  // namespace tl
