// fbn_sepsets.cu -- the separating sets of a learnt skeleton (Algorithm 1,
// SepSet) compacted on the device into CSR form: the removed pairs i < j in
// ascending (i, j), one offset per pair, the members in pair order.  The
// writer's outputs may be pinned host memory (device-addressable): only the
// compact arrays cross to the host.  Every kernel takes a batch of skeletons
// (grid.y), whose descriptors go by value: the export of 20 problems was 100
// launches and copies.
#include <cstdint>
#include <cuda_runtime.h>

#include "fbn_sepsets.h"

namespace fbn {
namespace {

constexpr int kSepJobs = 32;   // skeletons per launch
struct SepJobs {
    SepJob j[kSepJobs];
};

// Per row i (one warp): removed pairs (i, j > i) and their member total.
__global__ void k_sep_count(const __grid_constant__ SepJobs jobs)
{
    const SepJob& q = jobs.j[blockIdx.y];
    const int n = q.n;
    const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (i >= n) return;
    long long pairs = 0, members = 0;
    for (int j = i + 1 + lane; j < n; j += 32) {
        const int32_t L = q.sep_len[(long long)i * n + j];
        if (L >= 0) {
            pairs += 1;
            members += L;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
        members += __shfl_xor_sync(0xffffffffu, members, o);
    }
    if (lane == 0) {
        q.cnt[i] = pairs;
        q.cnt[n + i] = members;
    }
}

// One CTA per skeleton: exclusive row offsets of pairs and members, in place;
// the totals.
__global__ void k_sep_scan(const __grid_constant__ SepJobs jobs)
{
    const SepJob& q = jobs.j[blockIdx.x];
    const int n = q.n;
    long long* cnt = q.cnt;
    __shared__ long long sp[1024], sm[1024];
    const int t = threadIdx.x, T = blockDim.x;
    const int per = (n + T - 1) / T;
    const int lo = t * per, hi = lo + per < n ? lo + per : n;
    long long p = 0, m = 0;
    for (int i = lo; i < hi; ++i) {
        p += cnt[i];
        m += cnt[n + i];
    }
    sp[t] = p;
    sm[t] = m;
    __syncthreads();
    for (int o = 1; o < T; o <<= 1) {   // inclusive Hillis-Steele scan of the thread sums
        const long long ap = t >= o ? sp[t - o] : 0, am = t >= o ? sm[t - o] : 0;
        __syncthreads();
        sp[t] += ap;
        sm[t] += am;
        __syncthreads();
    }
    long long bp = sp[t] - p, bm = sm[t] - m;
    for (int i = lo; i < hi; ++i) {
        const long long cp = cnt[i], cm = cnt[n + i];
        cnt[i] = bp;
        cnt[n + i] = bm;
        bp += cp;
        bm += cm;
    }
    if (t == T - 1) {
        q.tot[0] = sp[T - 1];
        q.tot[1] = sm[T - 1];
    }
}

// Per row i (one warp): the row's pairs, offsets and members at its offsets.
__global__ void k_sep_write(const __grid_constant__ SepJobs jobs)
{
    const SepJob& q = jobs.j[blockIdx.y];
    const int n = q.n;
    const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (i >= n) return;
    long long p = q.cnt[i], m = q.cnt[n + i];
    for (int j0 = i + 1; j0 < n; j0 += 32) {
        const int j = j0 + lane;
        const int32_t L = j < n ? q.sep_len[(long long)i * n + j] : -1;
        const bool take = L >= 0;
        const unsigned ballot = __ballot_sync(0xffffffffu, take);
        long long inc = take ? L : 0;   // inclusive scan of the lengths
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (take) {
            const long long k = p + __popc(ballot & ((1u << lane) - 1u));
            const long long mo = m + inc - L;
            reinterpret_cast<int2*>(q.pairs)[k] = make_int2(i, j);
            q.offs[k] = mo;
            if (L > 0) {
                const int32_t* src = q.pool + q.sep_off[(long long)i * n + j];
                for (int t = 0; t < L; ++t) q.members[mo + t] = src[t];
            }
        }
        p += __popc(ballot);
        m += __shfl_sync(0xffffffffu, inc, 31);
    }
}

}  // namespace

// Launches kern over the jobs, rows of up to 8 per CTA on grid.x.
template <class K>
cudaError_t each_batch(K kern, const SepJob* jobs, int k, bool rows, int threads, cudaStream_t st)
{
    for (int at = 0; at < k; at += kSepJobs) {
        SepJobs a{};
        const int m = k - at < kSepJobs ? k - at : kSepJobs;
        int max_n = 1;
        for (int t = 0; t < m; ++t) {
            a.j[t] = jobs[at + t];
            max_n = jobs[at + t].n > max_n ? jobs[at + t].n : max_n;
        }
        const dim3 grid = rows ? dim3((max_n + 7) / 8, m) : dim3(m);
        kern<<<grid, threads, 0, st>>>(a);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_sep_count(const SepJob* jobs, int k, cudaStream_t st)
{
    const cudaError_t e = each_batch(k_sep_count, jobs, k, true, 256, st);
    return e != cudaSuccess ? e : each_batch(k_sep_scan, jobs, k, false, 1024, st);
}

cudaError_t launch_sep_write(const SepJob* jobs, int k, cudaStream_t st)
{
    return each_batch(k_sep_write, jobs, k, true, 256, st);
}

}  // namespace fbn
