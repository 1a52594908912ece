// fbn_pool_small.cu -- the small-table work-pool kernel (byte histograms).
#include "fbn_pool.cuh"

namespace fbn {

// Small-table class: the group size k_scan chose for this depth.
//
// What bounded it: instruction fetch (a counting loop per strategy, row count
// and group size, and 2,500 instructions of set-up, folding, marginals and
// logarithms around them: 3.3 of 14 stall cycles) and the latency of the sample
// rows (L1 hits 1%).  Now one counting loop for every copy count, the statistic
// from the n ln n table (a tenth of the instructions of FP32 terms), two
// vectors of every row in flight.  Two CTAs of 128 registers and 64 KB per SM:
// the rest of the SM's shared memory is the L1 the rows come through (100 KB:
// 2.6 ms at depth 2 of 256 problems, 72 KB 2.31, 64 KB 2.29, 48 KB 2.27 but 32%
// slower at the depths whose tables then miss a warp's slice).  Measured, test
// windows of depths 2 to 8 of 256 problems: 3.0 2.1 1.73 0.75 0.56 0.57 0.34 ->
// 2.3 1.28 1.12 0.53 0.26 0.08 0.03 ms; 1,000 variables x 100,000 samples, depths
// 2 to 4: 0.56 0.57 0.43 -> 0.39 0.34 0.42 ms.
__global__ void __launch_bounds__(kTestThreads, 2) k_pool_small(PoolArgs a)
{
    pdl_enter();
    extern __shared__ __align__(16) int smem[];
    __shared__ PoolShared sh;
    if (!a.ctr->active) return;
    switch (a.ctr->gsel) {
        case 32: pool_body<32>(a, smem, sh); break;
        case 64: pool_body<64>(a, smem, sh); break;
        case 128: pool_body<128>(a, smem, sh); break;
        default: pool_body<kTestThreads>(a, smem, sh); break;
    }
    tests_done(a.ctr);
}

}  // namespace fbn
