// fbn_sepsets.h -- host launchers of the separating-set compaction (fbn_sepsets.cu).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace fbn {

// One skeleton's separating sets and where their CSR form goes.  tot, pairs,
// offs and members may be device or device-addressable pinned host memory.
struct SepJob {
    const int32_t* sep_len;   // [n][n]
    const int64_t* sep_off;   // [n][n]
    const int32_t* pool;      // members at the pairs' offsets
    int n;
    long long* cnt;           // [2][n] device: row counts, then exclusive row offsets, of pairs and members
    long long* tot;           // [2] pairs and members in all
    int32_t* pairs;           // [R][2] (i < j, ascending), 8-byte aligned
    int64_t* offs;            // [R] (offs[R] is left to the caller)
    int32_t* members;
};

// Row offsets and totals of every job; then the CSR arrays.
cudaError_t launch_sep_count(const SepJob* jobs, int k, cudaStream_t st);
cudaError_t launch_sep_write(const SepJob* jobs, int k, cudaStream_t st);

}  // namespace fbn
