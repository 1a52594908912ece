// fbn_pool_marg.cu -- the kernels of depths 0 and 1 from one-hot planes.
#include "fbn_pool_marg.cuh"

namespace fbn {

__global__ void __launch_bounds__(kMargThreads, 2) k_pool_marg(PoolArgs a)
{
    pdl_enter();
    if (!a.ctr->active) return;
    marg_body<false>(a);
    tests_done(a.ctr);
}

__global__ void __launch_bounds__(kTestThreads) k_pairs_popc(const ProblemDev* probs, const int32_t* vtx_prob,
                                                             const int32_t* vtx_first, int total_vertices, int max_n,
                                                             const uint8_t* owned, PoolArgs a)
{
    pdl_enter();
    if (!a.ctr->active) return;
    pairs_popc_body<false>(probs, vtx_prob, vtx_first, total_vertices, max_n, owned, a);
    tests_done(a.ctr);
}

}  // namespace fbn
