// fbn_pool_big.cu -- the big-table work-pool kernel (CTA groups).
#include "fbn_pool.cuh"

namespace fbn {

// Big-table class: one CTA of 1,024 threads per test.  The class holds few
// tests of many cells (more than 16,384 by their bound), so what it costs is the
// latency of walking one table: with 256 threads per test the last two depths
// of 256 problems (118 and 9 tests) took 0.57 and 0.34 ms, now 0.08 and 0.03.
__global__ void __launch_bounds__(kBigThreads, 1) k_pool_big(PoolArgs a)
{
    pdl_enter();
    extern __shared__ __align__(16) int smem[];
    __shared__ PoolShared sh;
    if (!a.ctr->active || !a.ctr->wide) return;
    pool_body<kBigThreads>(a, smem, sh);
    tests_done(a.ctr);
}

}  // namespace fbn
