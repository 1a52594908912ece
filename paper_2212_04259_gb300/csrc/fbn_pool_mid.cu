// fbn_pool_mid.cu -- the big-table work-pool kernel for many tests (CTA groups).
#include "fbn_pool.cuh"

namespace fbn {

// The big-table class when its decision needs marginals (X^2, the observed df, or
// more samples than the n ln n table holds) and its tests are more than k_pool_big
// runs at once (DepthCounters::wide, see choose_pool).  Marginals and FP32 terms are
// chains of short phases behind barriers: two CTAs of 256 threads per SM cover one
// another's, where one of 1,024 waits.  X^2 with the observed df, depth 3 of 40
// variables of 6 values x 50,000 samples (13 M tests of 7,776 cells): 2,807 ms on
// k_pool_big, 1,230 here; X^2, depth 2 of 20 variables of 12 values (58,140 tests of
// 20,736 cells) 11.3 and 8.7 ms; depth 1 of 30 variables of 20 values 5.2 and 2.3.
__global__ void __launch_bounds__(kTestThreads, 2) k_pool_mid(PoolArgs a)
{
    pdl_enter();
    extern __shared__ __align__(16) int smem[];
    __shared__ PoolShared sh;
    if (!a.ctr->active || a.ctr->wide) return;
    pool_body<kTestThreads>(a, smem, sh);
    tests_done(a.ctr);
}

}  // namespace fbn
