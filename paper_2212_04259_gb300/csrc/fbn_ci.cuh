// fbn_ci.cuh -- one explicit CI test on a thread-block cluster (fbn_ci_test,
// fbn_ci_table, fbn_ci_test_noalloc): exact FP64 statistic and p-value
// (Section III-B).
//
// What bounds a single test is not memory (4 rows of 100,000 samples are
// 0.4 MB) but the latency of one SM: its sample loop, and above all the FP64
// statistic, whose logarithms run at 1/64 of the FP32 rate (a table of 3,000
// cells kept one SM busy for 70 us).  So a test runs on a cluster of up to 16
// CTAs.  Each CTA counts its share of the samples into its own table; the CTAs
// then split the strata of the conditioning set (a stratum's marginals and
// terms need no other stratum), each adding its strata's cells over the peers'
// tables through distributed shared memory; CTA 0 adds the partial statistics
// in rank order and its first warp evaluates the p-value, 32 terms of the sum
// at a time.  Tables over the shared-memory budget are counted into one global
// table by every CTA and reduced the same way.
#pragma once

#include <cmath>
#include <cooperative_groups.h>

#include "fbn_device.cuh"

namespace fbn {

constexpr int kCiMaxCluster = 16;     // non-portable cluster size (one GPC)
constexpr int kCiPortableCluster = 8;

// One explicit test, passed by value (no descriptor copy before the launch).
struct CiArgs {
    const uint8_t* rows[kMaxRows];    // S rows, X, Y
    uint8_t rad[kMaxRows];
    int nrows, rx, ry, N;
    long long cells;
    int* gtab;                        // global table of 3 * cells + 64 ints when the shared one does not fit
    double* out;                      // 3 doubles: statistic, df, p; nullptr: the table only
    int32_t* table_out;               // nullable
    unsigned* status;                 // nullable: receives the status bits
    double lgamma_a;                  // ln Gamma(df / 2) of the declared df
    int smem_ints, stat, df_mode;
};

// ln Gamma(df / 2) of the declared degrees of freedom, on the host.
inline double ci_lgamma(int rx, int ry, long long cells)
{
    int sign = 0;
    return lgamma_r(0.5 * (double)(rx - 1) * (double)(ry - 1) * (double)(cells / (rx * ry)), &sign);
}

// CTAs of a test: one per 4,096 samples (one 16-sample vector per thread) or
// per 96 cells of FP64 terms, whichever asks for more.  Measured per call, one
// CTA against this rule: tests of 100,003 samples with 0 to 3 conditioning
// variables 64 -> 32 us (16 CTAs), the table of 4 conditioning variables over
// 200,000 samples 143 -> 27 us (16 CTAs; the table alone skips the statistic).
inline int ci_cluster(long long N, long long cells, int max_cluster)
{
    const long long want = N / 4096 > cells / 96 ? N / 4096 : cells / 96;
    int k = 1;
    while (k < max_cluster && k < want) k *= 2;
    return k;
}

// Q(df/2, g2/2) by the CTA's first two warps, for integer df (both call; thread
// 0 gets the result).  Below the mean the series for P (A&S 6.5.29); above it
// the finite sum for integer df (A&S 26.4.4 and 26.4.5), from its largest term
// down: e^-x x^(a-1) / Gamma(a) (1 + (a-1)/x + (a-1)(a-2)/x^2 + ...), plus
// erfc(sqrt x) when df is odd.  All terms are positive.  Warp 0 adds the sum: each
// round takes 32 factors, one division per lane, and forms the 32 terms as a
// prefix product, where one thread's recurrence would wait for 32 dependent
// divisions.  Warp 1 evaluates the factor and erfc meanwhile: a dependent FP64
// operation takes some 100 cycles here, and the two chains are equally long
// (8 tests of 100,003 samples, one after the other: 260 us with both on one
// warp, 247 us so).
__device__ __forceinline__ double chisq_q_warps(double df, double g2, double lgamma_a, unsigned* status, double* share)
{
    const int lane = threadIdx.x & 31;
    const double a = 0.5 * df, x = 0.5 * g2;
    const bool lower = x < a + 1.0;
    if (!(g2 > 0.0)) return 1.0;   // the same for both warps
    if (threadIdx.x >= 32) {
        if (lane == 0) {
            share[0] = exp(a * log(x) - x - lgamma_a);   // x^a e^-x / Gamma(a)
            share[1] = !lower && fmod(df, 2.0) != 0.0 ? erfc(sqrt(x)) : 0.0;
        }
        asm volatile("bar.sync 1, 64;" ::: "memory");
        return 0.0;
    }
    const double kEps = 5e-16;
    const int kMaxRounds = 1 << 15;
    double carry = lower ? 1.0 / a : (a < 1.0 ? 0.0 : 1.0);   // the last term so far
    double sum = carry;
    int it = 0;
    for (; it < kMaxRounds; ++it) {
        const double j = (double)(it * 32 + lane + 1);
        double t = lower ? x / (a + j) : (a - j < 1.0 ? 0.0 : (a - j) / x);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double u = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t *= u;
        }
        t *= carry;
        carry = __shfl_sync(0xffffffffu, t, 31);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        sum += t;
        if (!(carry > sum * kEps)) break;
    }
    if (it == kMaxRounds && lane == 0) atomicOr(status, kStatusNumeric);
    asm volatile("bar.sync 1, 64;" ::: "memory");
    const double q = lower ? 1.0 - sum * share[0] : sum * (share[0] / x) + share[1];
    return q < 0.0 ? 0.0 : q > 1.0 ? 1.0 : q;
}

// Whether some sample value of the test's rows is not below its variable's
// arity (block-wide, every thread gets the answer): 16 samples per 16-byte
// load, four byte comparisons per 32-bit word.
__device__ __forceinline__ bool rows_out_of_range(const TestSpec& s)
{
    bool bad = false;
    const int nvec = s.N >> 4;
    for (int k0 = 0; k0 < s.nrows; k0 += 4) {   // four rows' loads in flight together: the check took 2.8 us of 15
        const int m = min(4, s.nrows - k0);
        for (int v = threadIdx.x; v < nvec; v += blockDim.x) {
            uint4 w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                w[k] = k < m ? __ldg(reinterpret_cast<const uint4*>(s.rows[k0 + k]) + v) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const unsigned rr = (k < m ? (unsigned)s.rad[k0 + k] : 255u) * 0x01010101u;   // the arity in each byte
                bad |= (__vcmpgeu4(w[k].x, rr) | __vcmpgeu4(w[k].y, rr) | __vcmpgeu4(w[k].z, rr) |
                        __vcmpgeu4(w[k].w, rr)) != 0u;
            }
        }
    }
    for (int t = (nvec << 4) + threadIdx.x; t < s.N; t += blockDim.x)
        for (int k = 0; k < s.nrows; ++k) bad |= s.rows[k][t] >= s.rad[k];
    return __syncthreads_or(bad) != 0;
}

// Shared-memory ints a CTA's share of the strata takes: cells and marginals,
// rounded to 16 bytes (the CTA's own table follows).
__host__ __device__ __forceinline__ long long ci_share_ints(long long cells, int rx, int ry, int k)
{
    const long long nz = cells / (rx * ry);
    return ((nz + k - 1) / k * (rx * ry + rx + ry + 1) + 3) / 4 * 4;
}

// Whether the test's table runs in shared memory on k CTAs.
__host__ __device__ __forceinline__ bool ci_fits_smem(long long cells, int rx, int ry, int k, long long smem_ints)
{
    const long long marg = cells / (rx * ry) * (rx + ry + 1);
    return cells + marg + (k > 1 ? ci_share_ints(cells, rx, ry, k) : 0) <= smem_ints;
}

// CHECK: the rows hold unvalidated values; a value out of range makes every
// output NaN and leaves the table unwritten.
template <bool CHECK>
__device__ __forceinline__ void ci_cluster_test(const CiArgs& q)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int k = (int)cl.num_blocks(), r = (int)cl.block_rank();
    extern __shared__ __align__(16) int smem[];
    __shared__ TestSpec spec;
    __shared__ double red[32];
    __shared__ double share[2];   // warp 1's half of the p-value (not red: warp 0 may still be adding up the statistic there)
    __shared__ double part[kCiMaxCluster], part_df[kCiMaxCluster];   // CTA 0: every CTA's share
    __shared__ int t_off, s_bad;
    __shared__ unsigned s_status;
    const int tid = threadIdx.x;
    // 16-sample boundaries: whole vectors of the rows
    const int lo = (int)((long long)q.N * r / k) & ~15;
    const int hi = r == k - 1 ? q.N : (int)((long long)q.N * (r + 1) / k) & ~15;
    if (tid < q.nrows) {
        spec.rows[tid] = q.rows[tid] + lo;
        spec.rad[tid] = q.rad[tid];
    }
    if (tid == 0) {
        spec.nrows = q.nrows;
        spec.rx = q.rx;
        spec.ry = q.ry;
        spec.N = hi - lo;
        spec.cells = q.cells;
        s_status = 0;
    }
    __syncthreads();
    if (CHECK) {
        const bool bad = rows_out_of_range(spec);
        if (k > 1) {   // out of range anywhere: known to every CTA before any counts
            if (tid == 0) s_bad = bad;
            cl.sync();
            const bool any = __syncthreads_or(tid < k && *cl.map_shared_rank(&s_bad, tid)) != 0;
            if (any) {
                if (r == 0 && tid == 0 && q.out) q.out[0] = q.out[1] = q.out[2] = nan("");
                cl.sync();   // no CTA leaves while a peer reads its flag
                return;
            }
        } else if (bad) {
            if (tid == 0 && q.out) q.out[0] = q.out[1] = q.out[2] = nan("");
            return;
        }
    }
    const int rxy = q.rx * q.ry;
    const int nz = (int)(q.cells / rxy);
    const int z0 = (int)((long long)nz * r / k), z1 = (int)((long long)nz * (r + 1) / k);
    const int c0 = z0 * rxy, c1 = z1 * rxy;
    int* T;          // this CTA's strata, summed over every CTA
    int* M;          // their marginals
    if (ci_fits_smem(q.cells, q.rx, q.ry, k, q.smem_ints)) {
        const long long share = k > 1 ? ci_share_ints(q.cells, q.rx, q.ry, k) : 0;
        int* own = grp_table<kTestThreads>(spec, smem + share, q.smem_ints - share, nullptr, 0, true, &M);
        T = own;
        if (k > 1) {
            if (tid == 0) t_off = (int)(own - smem);
            cl.sync();   // every table counted
            const int* peer[kCiMaxCluster];
#pragma unroll
            for (int p = 0; p < kCiMaxCluster; ++p)
                if (p < k) peer[p] = cl.map_shared_rank(smem, p) + *cl.map_shared_rank(&t_off, p);
            T = smem;
            M = smem + (c1 - c0);
            for (int c = c0 + tid; c < c1; c += kTestThreads) {
                int s = 0;
#pragma unroll
                for (int p = 0; p < kCiMaxCluster; ++p)
                    if (p < k) s += peer[p][c];
                T[c - c0] = s;
            }
        }
    } else {   // one global table, every CTA's samples
        for (int c = c0 + tid; c < c1; c += kTestThreads) q.gtab[c] = 0;
        __threadfence();
        if (k > 1) cl.sync(); else __syncthreads();
        count_global(spec, q.gtab, tid, kTestThreads);
        __threadfence();
        if (k > 1) cl.sync(); else __syncthreads();
        __threadfence();
        T = q.gtab + c0;
        const long long marg = (long long)(z1 - z0) * (q.rx + q.ry + 1);
        M = marg <= q.smem_ints ? smem : q.gtab + q.cells + (long long)z0 * (q.rx + q.ry + 1);
    }
    __syncthreads();
    if (q.table_out)
        for (int c = tid; c < c1 - c0; c += kTestThreads) q.table_out[c0 + c] = T[c];
    double st = 0.0, df = 0.0;
    if (q.out) {
        if (tid == 0) spec.cells = c1 - c0;   // the strata of this CTA from here on
        __syncthreads();
        if (c1 > c0) {
            grp_marginals<kTestThreads>(spec, T, M);
            st = q.stat == kStatX2 ? grp_x2_exact<kTestThreads>(spec, T, M, red)
                                   : grp_g2_exact<kTestThreads>(spec, T, M, red);
            if (q.df_mode) {
                __syncthreads();
                df = (double)grp_df_adjusted<kTestThreads>(spec, M, red);
            }
        }
    }
    if (k > 1) {   // also: no CTA leaves while a peer reads its table
        if (q.out && tid == 0) {
            *cl.map_shared_rank(&part[r], 0) = st;
            *cl.map_shared_rank(&part_df[r], 0) = df;
        }
        cl.sync();
        if (r != 0 || !q.out) return;
        st = df = 0.0;
        for (int p = 0; p < k; ++p) {
            st += part[p];
            df += part_df[p];
        }
    }
    if (!q.out || tid >= 64) return;
    double lg = q.lgamma_a;
    if (q.df_mode) lg = df > 0.0 ? lgamma(0.5 * df) : 0.0;
    else df = (double)(q.rx - 1) * (double)(q.ry - 1) * (double)nz;
    const double p = df > 0.0 ? chisq_q_warps(df, st, lg, &s_status, share) : 1.0;
    __syncwarp();
    if (tid == 0) {
        q.out[0] = st;
        q.out[1] = df;
        q.out[2] = !q.status && s_status ? nan("") : p;
        if (q.status) *q.status = s_status;
    }
}

// Largest cluster the kernel runs with on the current device and shared-memory
// size, after raising the kernel's limits (call once per device or handle).
template <typename K>
cudaError_t ci_prepare(K kern, size_t smem, int* max_cluster)
{
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    *max_cluster = kCiPortableCluster;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = kCiMaxCluster;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(kCiMaxCluster);
        cfg.blockDim = dim3(kTestThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n > 0) *max_cluster = kCiMaxCluster;
    }
    cudaGetLastError();
    return cudaSuccess;
}

template <typename K>
cudaError_t ci_launch(K kern, const CiArgs& q, int k, size_t smem, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = k;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(k);
    cfg.blockDim = dim3(kTestThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, q);
}

}  // namespace fbn
