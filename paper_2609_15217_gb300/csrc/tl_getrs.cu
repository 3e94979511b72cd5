// tl_getrs.cu -- launches of the shared-memory solves with given factors
// (tl_getrs.cuh).
#include "tl_getrs.cuh"
#include "tl_handle.h"

namespace tl {
namespace {

// One thread per right-hand side or T = 8 lanes per system, where measured
// faster than the register kernels (us, register kernel -> this one).  From
// six right-hand sides on a thread each: n = 12, 400,000 systems interleaved,
// r = 6 944 -> 822, r = 12 1768 -> 1240; n = 27, 178,062, r = 6 3781 ->
// 2272; 200 systems, r = 6 47 -> 27.  Three to five right-hand sides leave
// too few threads per system once n is large: n = 20, 360,576, r = 3 2201 ->
// 1740, but n = 32, 154,194, 2595 -> 3327; below n = 12 they tie.  Up to
// n = 9 one thread's registers hold a system, so large batches stay there
// (n = 6, 400,000, r = 32 801 against 1123) except per system from n = 8 on
// (n = 8, r = 6 388 -> 294) and interleaved up to 16 right-hand sides, beyond
// which n = 9 loses at first (n = 9, 400,000, r = 6 399 -> 365, r = 16 965 ->
// 936; 200,000, r = 17 531 against 540; n = 8 still gains: r = 16 817 -> 755,
// 200,000, r = 32 854 against 752).  Few large systems with few right-hand sides
// are better with 16 lanes each (n = 32, 200 systems, r = 6 73 against 82).
bool thread_per_rhs(const tl_handle *h, int n, int nrhs, int layout, int64_t batch)
{
    const int64_t sms = h->sm_count;
    if (nrhs < 6) return nrhs >= 3 && n >= 12 && n <= (nrhs == 3 ? 20 : 24) && batch > 4 * sms;
    if (n >= 28 && nrhs < 12) return batch > 16 * sms;
    if (n >= 10) return true;
    if (n >= 8) return layout == TL_LAYOUT_PER_SYSTEM || nrhs <= 16 || batch <= 16 * sms;
    return n >= 4 && batch <= 16 * sms;
}

// One or two right-hand sides, interleaved (where the register kernels' row
// accesses do not coalesce), n >= 17: n = 20, 400,000 systems, 1097 -> 818;
// n = 32, 172,334, 1353 -> 1132.  Small batches stay with the register
// kernels (n = 20, 200 systems: 23 and 24).
bool rows_in_shared(const tl_handle *h, int n, int nrhs, int layout, int64_t batch)
{
    return layout == TL_LAYOUT_INTERLEAVED && nrhs <= 2 && n >= 17 && batch > 32 * h->sm_count;
}

}  // namespace

bool getrs_in_shared(const tl_handle *h, int n, int nrhs, int layout, int64_t batch)
{
    return thread_per_rhs(h, n, nrhs, layout, batch) || rows_in_shared(h, n, nrhs, layout, batch);
}

tl_status launch_getrs_shared(tl_handle *h, int n, int layout, SolveArgs &args, cudaStream_t stream)
{
    const bool inter = layout == TL_LAYOUT_INTERLEAVED;
    const bool rows = args.nrhs < 3;
    const void *kern;
    if (rows)
        kern = n <= 24 ? reinterpret_cast<const void *>(&k_getrs_rows<8, 3>)
                       : reinterpret_cast<const void *>(&k_getrs_rows<8, 4>);
    else
        kern = inter ? reinterpret_cast<const void *>(&k_getrs_rhs<kInterleaved>)
                     : reinterpret_cast<const void *>(&k_getrs_rhs<kPerSystem>);
    int limit = 0;
    const tl_status st = smem_opt_in(h, kern, &limit);
    if (st != TL_OK) return st;
    GetrsPlan plan{};
    if (!(rows ? getrs_rows_plan(n, limit, &plan)
               : getrs_rhs_plan(n, args.nrhs, args.batch, limit, h->smem_per_sm, h->smem_reserved, &plan)))
        return TL_ERR_UNSUPPORTED;
    const int64_t grid = (args.batch + plan.SB - 1) / plan.SB;
    if (grid > INT32_MAX) return TL_ERR_UNSUPPORTED;
    int nn = n;
    void *params[] = {&args, &nn, &plan.SB};
    const cudaError_t e = cudaLaunchKernel(kern, dim3(static_cast<unsigned>(grid)),
                                           dim3(static_cast<unsigned>(plan.block)), params, plan.smem, stream);
    return e == cudaSuccess ? TL_OK : fail_cuda(h, e);
}

}  // namespace tl
