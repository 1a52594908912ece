// fbn_gram.h -- host launchers of the tcgen05 one-hot Gram (fbn_gram.cu).
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "fbn_internal.cuh"

namespace fbn {

size_t gram_smem_bytes();
int gram_rows_padded(int M);
long long gram_samples_padded(long long N);
cudaError_t launch_onehot(const ProblemDev* probs, const int32_t* vtx_prob, const int32_t* vtx_first,
                          int total_vertices, const DepthCounters* ctr, cudaStream_t st);
cudaError_t launch_zero_pad(const ProblemDev* probs, int nprob, cudaStream_t st);
cudaError_t encode_onehot_map(void* map, const uint8_t* E, int Mp, long long K);
size_t tensor_map_bytes();
int gram_unit_slices(const long long* tiles, const long long* stages, int k, int num_sms);
int gram_chunks(long long K, int unit_slices);
cudaError_t launch_gram(const void* maps, const int4* units, int n_units, int unit_slices, const ProblemDev* probs,
                        int num_sms, unsigned* status, int wait_limit, cudaStream_t st);

// Pair tables (and, with ctr, the decisions of depth 0) from the Gram.
struct PairsGramArgs {
    int emit = 0;            // write the full tables
    int sym = 0;             // the transposed blocks and the zeros of the diagonal blocks too
    int32_t* out = nullptr;  // where (row stride ldo); nullptr: each problem's gram
    long long ldo = 0;
    long long total_pairs = 0;
    CritTableDev crit{};
    double alpha = 0.0;
    DepthCounters* ctr = nullptr;
    int stat = 0, df_mode = 0;
    int max_arity = 0;       // of the call
};
// Problems with a variable of more values than this go through k_pairs_wide, a launch of its own.
constexpr int kWideArity = 8;
cudaError_t launch_pairs_gram(const ProblemDev* probs, const int32_t* vtx_prob, const int32_t* vtx_first,
                              int total_vertices, int max_n, const PairsGramArgs& a, int num_sms, cudaStream_t st);

}  // namespace fbn
