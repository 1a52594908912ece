// fbn_ci.cu -- the explicit-test kernel of fbn_ci_test and fbn_ci_table (the
// test itself in fbn_ci.cuh).
#include "fbn_ci.cuh"
#include "fbn_launch.h"

namespace fbn {
namespace {

__global__ void __launch_bounds__(kTestThreads, 2) k_ci_test(const __grid_constant__ CiArgs q)
{
    ci_cluster_test<false>(q);
}

}  // namespace

cudaError_t prepare_ci(size_t smem_bytes, int* max_cluster)
{
    return ci_prepare(k_ci_test, smem_bytes, max_cluster);
}

cudaError_t launch_ci(const CiArgs& q, int cluster, size_t smem_bytes, cudaStream_t st)
{
    return ci_launch(k_ci_test, q, cluster, smem_bytes, st);
}

}  // namespace fbn
