// Block plans of the solves with given factors (tl_getrs_plan.h): for every n,
// number of right-hand sides and batch, and shared-memory limits from a few
// KiB up, a plan fits its limit and the kernel's block, holds whole systems,
// and is refused only when not even one system fits.
#include <cstdio>

#include "tl_getrs_plan.h"

static int fail(const char *what, int n, int nrhs, long long batch, size_t limit)
{
    std::printf("%s: n %d, nrhs %d, batch %lld, limit %zu\n", what, n, nrhs, batch, limit);
    return 1;
}

int main()
{
    const size_t limits[] = {2048, 8192, 48 * 1024, 101376, 232448};
    const long long batches[] = {1, 2, 3, 31, 128, 1000000};
    int refused = 0;
    for (int n = 1; n <= 32; ++n)
        for (size_t limit : limits) {
            tl::GetrsPlan p{};
            const size_t rows = static_cast<size_t>(tl::getrs_block_doubles(n, 8)) * 8;
            if (tl::getrs_rows_plan(n, limit, &p) != (rows <= limit)) return fail("rows", n, 1, 0, limit);
            for (int nrhs = 1; nrhs <= 32; ++nrhs)
                for (long long batch : batches) {
                    const int threads1 = (nrhs + 31) / 32 * 32;
                    const size_t one =
                        (static_cast<size_t>(tl::getrs_block_doubles(n, 1)) + static_cast<size_t>(n) * threads1) * 8;
                    // an SM of the block's own limit and one with room for more
                    for (size_t per_sm : {limit + 1024, limit * 2}) {
                        const bool ok = tl::getrs_rhs_plan(n, nrhs, batch, limit, per_sm, 1024, &p);
                        if (ok != (one <= limit)) return fail("refusal", n, nrhs, batch, limit);
                        if (!ok) {
                            ++refused;
                            continue;
                        }
                        const size_t need = (static_cast<size_t>(tl::getrs_block_doubles(n, p.SB)) +
                                             static_cast<size_t>(n) * p.block) * 8;
                        if (p.smem != need || p.smem > limit) return fail("bytes", n, nrhs, batch, limit);
                        if (p.block > 128 || p.block % 32 || p.SB < 1 || p.SB > batch || p.SB * nrhs > p.block)
                            return fail("block", n, nrhs, batch, limit);
                    }
                }
        }
    if (!refused) return fail("nothing refused", 0, 0, 0, 0);
    std::puts("ok");
    return 0;
}
