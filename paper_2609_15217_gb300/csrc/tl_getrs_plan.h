// tl_getrs_plan.h -- shared memory and block shape of the solves with given
// factors (tl_getrs.cuh).  Pure C++ on the host side, no CUDA calls.
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>

#ifdef __CUDACC__
#define TL_HOST_DEVICE __host__ __device__
#else
#define TL_HOST_DEVICE
#endif

namespace tl {

// One system in shared memory: n rows of n entries (odd stride), n
// reciprocals, n pivots and n source rows of P (int32); an odd number of
// doubles, so that the systems of a warp start on distinct banks.
TL_HOST_DEVICE constexpr int getrs_row_stride(int n) { return n | 1; }
TL_HOST_DEVICE constexpr int getrs_sys_doubles(int n) { return (n * getrs_row_stride(n) + 2 * n) | 1; }
// Doubles of a block of SB systems: theirs and a flag each.
TL_HOST_DEVICE constexpr int getrs_block_doubles(int n, int SB) { return SB * getrs_sys_doubles(n) + (SB + 1) / 2; }

struct GetrsPlan {
    int SB;       // systems per block
    int block;    // threads
    size_t smem;  // bytes of dynamic shared memory
};

// k_getrs_rhs: the systems per block that keep the most useful lanes on an
// SM, up to the two warps per sub-partition that keep the FP64 pipe busy.
// `limit`: dynamic shared memory a block may use; `per_sm`: shared memory of
// an SM, of which every block also takes `reserved`.  False when not even one
// system fits.
inline bool getrs_rhs_plan(int n, int nrhs, int64_t batch, size_t limit, size_t per_sm, size_t reserved, GetrsPlan *plan)
{
    double best = -1.0;
    const int most = static_cast<int>(std::min<int64_t>(128 / nrhs, batch));
    for (int sb = 1; sb <= most; ++sb) {
        const int threads = (sb * nrhs + 31) / 32 * 32;
        const size_t bytes = (static_cast<size_t>(getrs_block_doubles(n, sb)) + static_cast<size_t>(n) * threads) * 8;
        if (bytes > limit) break;
        const int blocks = static_cast<int>(per_sm / (bytes + reserved));
        const int warps = std::min(8, blocks * threads / 32);
        const double score = warps * static_cast<double>(sb * nrhs) / threads;
        if (score >= best) {
            best = score;
            *plan = GetrsPlan{sb, threads, bytes};
        }
    }
    return best >= 0.0;
}

// k_getrs_rows: 8 systems of 8 lanes in a block.
inline bool getrs_rows_plan(int n, size_t limit, GetrsPlan *plan)
{
    *plan = GetrsPlan{8, 64, static_cast<size_t>(getrs_block_doubles(n, 8)) * 8};
    return plan->smem <= limit;
}

}  // namespace tl
