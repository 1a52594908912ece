// fbn_gram.cu -- depth 0 of Algorithm 1 as a one-hot Gram product on the
// fifth-generation tensor cores of sm_103a (tcgen05), all pairs at once.
//
// For every variable v and value x let e_{v,x} in {0,1}^N mark the samples
// with V_v = x.  The depth-0 contingency table of the pair (i, j) is
// N_ij(x, y) = <e_{i,x}, e_{j,y}>, so all n(n-1)/2 tables (Section IV-B: depth
// zero tests every pair of the complete graph once) are blocks of a Gram matrix
// E E^T of one-hot rows.  Only the rows of the values >= 1 are multiplied: the
// diagonal holds the counts of single values, and every cell of value 0 follows
// from them.  For arities 2 to 5 that halves the products (rows 3,500 -> 2,500
// for 1,000 variables) and cuts the operand by 0.71.
//
// E is built in HBM as FP8 E4M3 (0 and 1 are exact).  The product runs on
// tcgen05.mma.kind::f8f6f4 with FP32 accumulators in tensor memory; every
// accumulation covers at most kChunk = 8192 samples, so each partial sum is an
// integer below 2^13 and exact even if the accumulation kept only 14
// significant bits.  Each chunk's 128x256 tile is added into an INT32 Gram in
// global memory.  (tcgen05.mma.kind::i8 does not assemble for sm_103a with this
// toolkit, hence FP8 0/1 operands.)
//
// A tile is 128 rows of E against 256 rows (M = 128, N = 256 per MMA): each
// 128-sample stage brings 48 KB of operands for 8 MFLOP, a third less operand
// traffic per FLOP than square 128-row tiles.  Work unit = (128-row tile,
// 256-row tile reaching the upper triangle, chunk of samples), chunk-major so
// that the CTAs of a wave stream the same sample range and share it in L2.
// CTA roles: warps 0-3 epilogue (TMEM -> registers -> coalesced INT32 atomic
// adds), warp 4 TMA producer, warp 5 MMA issuer and TMEM owner.
#include <algorithm>
#include <cstdint>

#include <cuda.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include "fbn_depth.cuh"
#include "fbn_gram.h"
#include "fbn_tc.cuh"

namespace fbn {
namespace {

using namespace tc;

constexpr int kTile = 128;                           // rows of an A tile = M of one MMA
constexpr int kTileN = 256;                          // rows of a B tile = N of one MMA
constexpr int kKSlice = 128;                         // samples (bytes) per pipeline stage
constexpr int kChunk = 8192;                         // samples per exact accumulation
constexpr int kSlicesPerChunk = kChunk / kKSlice;
constexpr int kStages = 4;
constexpr int kEpilogueStages = 48;                  // a unit's epilogue in stages (gram_unit_slices)
constexpr int kTileBytes = kTile * kKSlice;          // 16 KB
constexpr int kStageBytes = 3 * kTileBytes;          // A + the two 128-row halves of B
constexpr int kGramThreads = 192;
constexpr uint32_t kTmemCols = 512;                  // two 256-column FP32 accumulators
constexpr int kStagePad = 33;                        // epilogue transpose tile row (ints)
constexpr size_t kGramSmem = 1024 /*align*/ + (size_t)kStages * kStageBytes + 4 * 32 * kStagePad * 4 + 256;

constexpr uint32_t kIdesc = tc::idesc_f8(kTile, kTileN);

// Work unit of the Gram: problem, 128-row tile ti, 256-row tile tj covering
// some column >= some row (tj >= ti / 2), chunk of samples.
struct GramArgs {
    const CUtensorMap* maps;    // [problems] tensor maps of the one-hot matrices (global memory)
    const int4* units;          // [n_units] (problem, ti, tj, chunk)
    const ProblemDev* probs;
    int n_units;
    int unit_slices;            // stages per work unit, at most kSlicesPerChunk (exact accumulation)
    unsigned* status;
    unsigned limit;             // attempts of each role's bounded wait
};

__global__ void __launch_bounds__(kGramThreads, 1) k_gram(GramArgs g)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    int* xpose = reinterpret_cast<int*>(smem + (size_t)kStages * kStageBytes);          // 4 x 32 x 33 ints
    uint64_t* bars = reinterpret_cast<uint64_t*>(xpose + 4 * 32 * kStagePad);
    uint64_t* full = bars;                 // [kStages] TMA -> MMA
    uint64_t* empty = bars + kStages;      // [kStages] MMA -> TMA
    uint64_t* acc_full = bars + 2 * kStages;       // [2] MMA -> epilogue
    uint64_t* acc_empty = bars + 2 * kStages + 2;  // [2] epilogue -> MMA
    uint64_t* drain = bars + 2 * kStages + 4;      // MMA completion before teardown
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 5);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    int* issued = reinterpret_cast<int*>(tmem_slot + 2);   // [kStages], producer thread only

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int U = g.n_units;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(smem_u32(&full[s]), 1);
            mbar_init(smem_u32(&empty[s]), 1);
            issued[s] = 0;
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&acc_full[b]), 1);
            mbar_init(smem_u32(&acc_empty[b]), 4);   // one arrive per epilogue warp
        }
        mbar_init(smem_u32(drain), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 5) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 4) {
        // ---------------- TMA producer
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            int fenced = -1;
            for (int u = blockIdx.x; u < U && !*abort_flag; u += gridDim.x) {
                const int4 t = g.units[u];
                const CUtensorMap* map = g.maps + t.x;
                if (t.x != fenced) {   // the host rewrites the maps between launches
                    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(map) : "memory");
                    fenced = t.x;
                }
                const int slices = (int)(g.probs[t.x].onehot_ld / kKSlice);
                const int kb0 = t.w * g.unit_slices;
                const int kb1 = min(kb0 + g.unit_slices, slices);
                for (int kb = kb0; kb < kb1; ++kb) {
                    if (!mbar_wait(smem_u32(&empty[stage]), phase ^ 1u, abort_flag, g.status, g.limit)) break;
                    const uint32_t fb = smem_u32(&full[stage]);
                    const uint32_t a = smem_u32(smem + (size_t)stage * kStageBytes);
                    mbar_expect_tx(fb, kStageBytes);
                    tma_load_2d(a, map, fb, kb * kKSlice, t.y * kTile);
                    // B: rows beyond the padded matrix (odd tile count) come back as zeros
                    tma_load_2d(a + kTileBytes, map, fb, kb * kKSlice, t.z * kTileN);
                    tma_load_2d(a + 2 * kTileBytes, map, fb, kb * kKSlice, t.z * kTileN + kTile);
                    issued[stage] += 1;
                    if (++stage == kStages) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
        }
    } else if (warp == 5) {
        // ---------------- MMA issuer (one thread)
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            int acc = 0;
            uint32_t acc_phase = 0;
            bool ok = true;
            for (int u = blockIdx.x; u < U && ok; u += gridDim.x) {
                const int4 t = g.units[u];
                const int slices = (int)(g.probs[t.x].onehot_ld / kKSlice);
                const int kb0 = t.w * g.unit_slices;
                const int kb1 = min(kb0 + g.unit_slices, slices);
                if (!mbar_wait(smem_u32(&acc_empty[acc]), acc_phase ^ 1u, abort_flag, g.status, g.limit)) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem + (uint32_t)(acc * kTileN);
                for (int kb = kb0; kb < kb1; ++kb) {
                    if (!mbar_wait(smem_u32(&full[stage]), phase, abort_flag, g.status, g.limit)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t a = smem_u32(smem + (size_t)stage * kStageBytes);
                    const uint64_t da = smem_desc(a), db = smem_desc(a + kTileBytes);
#pragma unroll
                    for (int k = 0; k < kKSlice / 32; ++k)   // 32 E4M3 values = 32 bytes of K per MMA
                        mma_f8(d_tmem, da + (uint64_t)(2 * k), db + (uint64_t)(2 * k), kIdesc, (kb > kb0 || k > 0) ? 1u : 0u);
                    mma_commit(smem_u32(&empty[stage]));
                    if (++stage == kStages) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
                if (!ok) break;
                mma_commit(smem_u32(&acc_full[acc]));
                acc ^= 1;
                if (acc == 0) acc_phase ^= 1u;
            }
            // every MMA this thread issued has finished before TMEM is released
            // (the default bound here, whatever the roles' bound)
            mma_commit(smem_u32(drain));
            for (unsigned it = 0; it < kSpinLimit; ++it)
                if (mbar_try(smem_u32(drain), 0)) break;
        }
    } else {
        // ---------------- epilogue: warps 0-3, TMEM lanes 32w .. 32w+31
        int* xp = xpose + warp * 32 * kStagePad;
        int acc = 0;
        uint32_t acc_phase = 0;
        for (int u = blockIdx.x; u < U; u += gridDim.x) {
            const int4 t = g.units[u];
            int32_t* G = g.probs[t.x].rgram;
            const long long ldg = g.probs[t.x].rgram_ld;
            if (!mbar_wait(smem_u32(&acc_full[acc]), acc_phase, abort_flag, g.status, g.limit)) break;
            tc_fence_after();
            const uint32_t base = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(acc * kTileN);
            const long long row0 = (long long)t.y * kTile + warp * 32;
            for (int j0 = 0; j0 < kTileN; j0 += 32) {
                if ((long long)t.z * kTileN + j0 >= ldg) break;   // columns past the padded matrix
                uint32_t v[32];
                tmem_ld32(base + (uint32_t)j0, v);
#pragma unroll
                for (int q = 0; q < 32; ++q) xp[lane * kStagePad + q] = __float2int_rn(__uint_as_float(v[q]));
                __syncwarp();
                int32_t* dst = G + row0 * ldg + (long long)t.z * kTileN + j0 + lane;
#pragma unroll 4
                for (int r = 0; r < 32; ++r) {
                    const int val = xp[r * kStagePad + lane];
                    if (val) atomicAdd(dst + (long long)r * ldg, val);
                }
                __syncwarp();
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&acc_empty[acc]));
            acc ^= 1;
            if (acc == 0) acc_phase ^= 1u;
        }
    }

    __syncthreads();
    if (warp == 4 && lane == 0) {
        // no TMA write may land after the CTA exits: wait for the last load of
        // every stage (immediate unless a role gave up)
        for (int s = 0; s < kStages; ++s)
            if (issued[s] > 0) {
                for (unsigned it = 0; it < kSpinLimit; ++it)
                    if (mbar_try(smem_u32(&full[s]), (uint32_t)((issued[s] - 1) & 1))) break;
            }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 5) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

// One-hot matrix E of every problem: row roff_v + x - 1, x >= 1, holds 0x38
// (E4M3 1.0) where V_v = x, else 0; samples at or beyond N (the padding of the store)
// are 0 for every row.  One CTA per variable of the batch.
// ctr: nullable; the depth whose tests start here.
__global__ void k_onehot(const ProblemDev* __restrict__ probs, const int32_t* __restrict__ vtx_prob,
                         const int32_t* __restrict__ vtx_first, int total_vertices, const DepthCounters* ctr)
{
    const int g = blockIdx.x;
    if (g >= total_vertices) return;
    if (ctr && g == 0 && threadIdx.x == 0)
        if (DepthRecord* r = depth_rec(ctr, ctr->d)) r->t_begin = r->t_tests = gtime();
    const int p = vtx_prob[g];
    const ProblemDev& P = probs[p];
    const int v = g - vtx_first[p];
    const int r = P.ar[v];
    const long long K = P.onehot_ld;
    const uint4* row = reinterpret_cast<const uint4*>(P.data + (long long)v * P.ld);
    uint8_t* E = P.onehot + (long long)P.roff[v] * K;
    const long long nvec = K / 16;
    for (long long q = threadIdx.x; q < nvec; q += blockDim.x) {
        const uint4 w = row[q];   // padding past the samples is value 0: no row
        for (int x = 1; x < r; ++x) {
            const uint32_t rep = 0x01010101u * (uint32_t)x;
            uint4 o;
            o.x = __vcmpeq4(w.x, rep) & 0x38383838u;
            o.y = __vcmpeq4(w.y, rep) & 0x38383838u;
            o.z = __vcmpeq4(w.z, rep) & 0x38383838u;
            o.w = __vcmpeq4(w.w, rep) & 0x38383838u;
            reinterpret_cast<uint4*>(E + (long long)(x - 1) * K)[q] = o;
        }
    }
}

// --------------------------------------------------------------------------
// From the Gram over the values >= 1 to every pair's table and decision.
//
// A warp takes one variable i and 32 consecutive j, one pair per lane: the
// lanes read neighbouring columns of i's Gram rows.  The cells of value 0
// follow from the single counts (the Gram's diagonal): N(x, 0) = N_i(x) - sum_y
// N(x, y), and so on.  At depth 0 the graph is complete, so the pairs need no
// edge list: the kernel writes the adjacency, the empty separating sets and the
// depth's counters itself, and (emit) the full tables that depth 1 reads its
// margins from.
struct PairGram {
    const ProblemDev* P;
    const int32_t* R;      // Gram rows of i, columns of j
    const int32_t *si, *sj;   // single counts of value 1 of i and j (diagonal), strides ldr + 1
    long long ldr;
    int ri, rj, N;

    __device__ __forceinline__ PairGram(const ProblemDev& p, int i, int j) : P(&p)
    {
        ldr = p.rgram_ld;
        const long long oi = p.roff[i], oj = p.roff[j];
        R = p.rgram + oi * ldr + oj;
        si = p.rgram + oi * (ldr + 1);
        sj = p.rgram + oj * (ldr + 1);
        ri = p.ar[i];
        rj = p.ar[j];
        N = p.N;
    }
    __device__ __forceinline__ int both(int x, int y) const { return R[(x - 1) * ldr + y - 1]; }   // x, y >= 1
    __device__ __forceinline__ int single_i(int x) const { return si[(x - 1) * (ldr + 1)]; }
    __device__ __forceinline__ int single_j(int y) const { return sj[(y - 1) * (ldr + 1)]; }
    // one cell on its own (the exact decision)
    __device__ int cell(int x, int y) const
    {
        if (x > 0 && y > 0) return both(x, y);
        if (x > 0) {
            int s = single_i(x);
            for (int b = 1; b < rj; ++b) s -= both(x, b);
            return s;
        }
        if (y > 0) {
            int s = single_j(y);
            for (int a = 1; a < ri; ++a) s -= both(a, y);
            return s;
        }
        int s = N;
        for (int b = 1; b < rj; ++b) s -= single_j(b);
        for (int a = 1; a < ri; ++a) {
            s -= single_i(a);
            for (int b = 1; b < rj; ++b) s += both(a, b);
        }
        return s;
    }
    __device__ int margin_i(int x) const
    {
        if (x > 0) return single_i(x);
        int s = N;
        for (int a = 1; a < ri; ++a) s -= single_i(a);
        return s;
    }
    __device__ int margin_j(int y) const
    {
        if (y > 0) return single_j(y);
        int s = N;
        for (int b = 1; b < rj; ++b) s -= single_j(b);
        return s;
    }
};

// The exact FP64 statistic of one pair by the whole warp (the pair of the lane
// whose FP32 band straddled crit).
__device__ __noinline__ double pair_stat_exact(const ProblemDev& P, int i, int j, int stat)
{
    const PairGram g(P, i, j);
    double st = 0.0;
    for (int c = threadIdx.x & 31; c < g.ri * g.rj; c += 32) {
        const int x = c / g.rj, y = c - x * g.rj;
        const int n = g.cell(x, y);
        const long long nx = g.margin_i(x), ny = g.margin_j(y);
        const long long p = (long long)n * g.N, q = nx * ny;
        if (stat == kStatX2) {
            if (q > 0) {
                const double dd = (double)(p - q);
                st += dd * dd / ((double)g.N * (double)nx * (double)ny);
            }
        } else if (n > 0) {
            st += 2.0 * (double)n * log1p((double)(p - q) / (double)q);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) st += __shfl_xor_sync(0xffffffffu, st, o);
    return st;
}

constexpr int kPairArity = 5;   // blocks of at most this many values a side are held in registers

// DECIDE: the depth-0 decisions into adj, sep_len, sep_off and the counters.
// emit: full tables into G with row stride ldg (0: the problem's gram), the
// transposed blocks too when sym.
template <bool DECIDE>
__global__ void __launch_bounds__(256) k_pairs_gram(const ProblemDev* __restrict__ probs,
                                                    const int32_t* __restrict__ vtx_prob,
                                                    const int32_t* __restrict__ vtx_first, int total_vertices,
                                                    int blocks_n, int emit, int sym, int32_t* G_out, long long ldg,
                                                    long long total_pairs, CritTableDev crit, double alpha,
                                                    DepthCounters* ctr, int stat, int df_mode)
{
    __shared__ int s_cell[8][kPairArity * kPairArity][32], s_nj[8][kPairArity][32];   // 8 warps: a column per lane
    const int lane = threadIdx.x & 31;
    if (DECIDE && !ctr->active) return;
    const long long tasks = (long long)total_vertices * blocks_n;
    const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
    unsigned long long removed = 0, samples = 0, tests = 0;
    for (long long t = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < tasks; t += warps) {
        const int g = (int)(t / blocks_n), j0 = (int)(t - (long long)g * blocks_n) * 32;
        const int p = vtx_prob[g];
        const ProblemDev& P = probs[p];
        const int i = g - vtx_first[p], n = P.n;
        if (j0 >= n || j0 + 31 < i) continue;
        const int j = j0 + lane;
        int32_t* G = emit ? (G_out ? G_out : P.gram) : nullptr;
        const long long ld = G_out ? ldg : P.gram_ld;
        const int oi = P.off[i];
        if (P.max_arity > kWideArity) continue;   // k_pairs_wide
        if (j == i) {   // the diagonal block
            const PairGram d(P, i, i);
            if (G)
                for (int x = 0; x < d.ri; ++x) {
                    if (sym)
                        for (int y = 0; y < d.ri; ++y) G[(oi + x) * ld + oi + y] = 0;
                    G[(oi + x) * (ld + 1)] = d.margin_i(x);
                }
            if (DECIDE) P.adj[(long long)i * n + i] = 0;
        }
        const bool pair = j > i && j < n;
        int dec = 0;
        long long df = 0;
        if (pair) {
            const PairGram q(P, i, j);
            const int ri = q.ri, rj = q.rj, N = q.N, oj = P.off[j];
            const bool narrow = N < 65536;
            float acc = 0.0f, mag = 0.0f;
            int ni0 = N, nj0 = N, ax = 0, ay = 0;
            auto put = [&](int x, int y, int v) {
                if (!G) return;
                G[(oi + x) * ld + oj + y] = v;
                if (sym) G[(oj + y) * ld + oi + x] = v;
            };
            auto term = [&](int v, int nx, int ny) {
                if (DECIDE && nx > 0 && ny > 0) marg_term(v, N, nx, ny, narrow, stat, acc, mag);
            };
            if (P.max_arity <= kPairArity) {
                // the block's loads in flight together, its cells through this
                // lane's column of shared memory, so that the terms are one
                // small loop (the loads still spill some 250 bytes of 128
                // registers in the deciding kernel)
                int (*cv)[32] = s_cell[threadIdx.x >> 5];
                int (*cj)[32] = s_nj[threadIdx.x >> 5];
                int v[kPairArity - 1][kPairArity - 1], nj[kPairArity - 1], ni[kPairArity - 1];
#pragma unroll
                for (int b = 0; b < kPairArity - 1; ++b) nj[b] = b + 1 < rj ? q.single_j(b + 1) : 0;
#pragma unroll
                for (int a = 0; a < kPairArity - 1; ++a) {
                    ni[a] = a + 1 < ri ? q.single_i(a + 1) : 0;
#pragma unroll
                    for (int b = 0; b < kPairArity - 1; ++b) v[a][b] = a + 1 < ri && b + 1 < rj ? q.both(a + 1, b + 1) : 0;
                }
#pragma unroll
                for (int b = 0; b < kPairArity - 1; ++b) {
                    nj0 -= nj[b];
                    ay += nj[b] > 0;
                    cj[b + 1][lane] = nj[b];
                }
                cj[0][lane] = nj0;
#pragma unroll
                for (int a = 0; a < kPairArity - 1; ++a) {
                    ni0 -= ni[a];
                    ax += ni[a] > 0;
                }
                int n00 = nj0;
#pragma unroll
                for (int a = 0; a < kPairArity - 1; ++a) {
                    int rest = ni[a];
#pragma unroll
                    for (int b = 0; b < kPairArity - 1; ++b) {
                        rest -= v[a][b];
                        nj[b] -= v[a][b];
                        cv[(a + 1) * kPairArity + b + 1][lane] = v[a][b];
                    }
                    n00 -= rest;
                    cv[(a + 1) * kPairArity][lane] = rest;
                }
#pragma unroll
                for (int b = 0; b < kPairArity - 1; ++b) cv[b + 1][lane] = nj[b];
                cv[0][lane] = n00;
                for (int x = 0; x < ri; ++x) {
                    const int nx = x ? q.single_i(x) : ni0;
                    for (int y = 0; y < rj; ++y) {
                        const int c = cv[x * kPairArity + y][lane];
                        put(x, y, c);
                        term(c, nx, cj[y][lane]);
                    }
                }
            } else {   // up to kWideArity: the block read twice
                for (int y = 1; y < rj; ++y) {
                    const int ny = q.single_j(y);
                    nj0 -= ny;
                    ay += ny > 0;
                }
                int n00 = nj0;
                for (int x = 1; x < ri; ++x) {
                    const int nx = q.single_i(x);
                    ni0 -= nx;
                    ax += nx > 0;
                    int rest = nx;
                    for (int y = 1; y < rj; ++y) {
                        const int v = q.both(x, y);
                        rest -= v;
                        put(x, y, v);
                        term(v, nx, q.single_j(y));
                    }
                    n00 -= rest;
                    put(x, 0, rest);
                    term(rest, nx, nj0);
                }
                for (int y = 1; y < rj; ++y) {
                    int v = q.single_j(y);
                    for (int x = 1; x < ri; ++x) v -= q.both(x, y);
                    put(0, y, v);
                    term(v, ni0, q.single_j(y));
                }
                put(0, 0, n00);
                term(n00, ni0, nj0);
            }
            ax += ni0 > 0;
            ay += nj0 > 0;
            if (DECIDE) {
                df = df_mode ? (long long)(ax - 1) * (ay - 1) : (long long)(ri - 1) * (rj - 1);
                if (df <= 0) {
                    dec = 1;   // p = 1 > alpha
                } else {
                    float2 f = make_float2(0.0f, 0.0f);
                    if (df < crit.dense_n) f = crit.dense_f[df];
                    if (!(f.y > 0.0f)) {
                        const double c = crit_get(crit, df, alpha, &ctr->status);
                        f = make_float2(__double2float_rd(c), __double2float_ru(c));
                    }
                    dec = decide_from_sums(acc, mag, (float)(ri * rj), 0.0f, stat, f.x, f.y, kMargTermRel);
                }
            }
        }
        if constexpr (DECIDE) {
            unsigned open = __ballot_sync(0xffffffffu, dec < 0);
            while (open) {   // the band straddles crit: exactly, one such pair at a time
                const int l = __ffs(open) - 1;
                open &= open - 1;
                const double st = pair_stat_exact(P, i, j0 + l, stat);
                if (lane == l) dec = st < crit_get(crit, df, alpha, &ctr->status);
                __syncwarp();
            }
            if (pair) {
                P.adj[(long long)i * n + j] = (uint8_t)(dec ? 0 : 1);
                P.adj[(long long)j * n + i] = (uint8_t)(dec ? 0 : 1);
                P.sep_len[(long long)i * n + j] = dec ? 0 : -1;
                P.sep_off[(long long)i * n + j] = 0;
                removed += dec != 0;
                tests += 1;
                samples += (unsigned long long)P.N;
            }
        }
    }
    if constexpr (DECIDE) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            removed += __shfl_xor_sync(0xffffffffu, removed, o);
            tests += __shfl_xor_sync(0xffffffffu, tests, o);
            samples += __shfl_xor_sync(0xffffffffu, samples, o);
        }
        if (lane == 0 && tests) {   // one test per pair
            atomicAdd(&ctr->removed, removed);
            atomicAdd(&ctr->tests, tests);
            atomicAdd(&ctr->tests_oracle, tests);
            atomicAdd(&ctr->test_samples, samples);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            if (blockIdx.x == 0) ctr->n_edges[0] = (unsigned long long)total_pairs;   // the depth's edges: every pair
            if (DepthRecord* r = depth_rec(ctr, ctr->d)) atomicMax(&r->t_tests_end, gtime());
        }
    }
}

// The same for problems with an arity above kWideArity: a group of G threads per pair
// (a warp up to 32 values, a CTA of 256 threads up to 64, of 1,024 above), its rows
// across the lanes, the decision in FP64.  One lane per pair walked a block alone and
// added the terms in FP32: pair counts on the device of 10 variables of 200 values x
// 3,000 samples 9.19 -> 0.11 ms, of 100 of 30 values x 20,000 0.49 -> 0.22 ms, depth 0
// of 40 of 255 values x 10,000 45.8 -> 6.2 ms.  FP64 costs where blocks are small:
// depth 0 of 300 variables of 10 values x 20,000 0.25 -> 0.65 ms.  (With 1,024 threads
// the deciding kernel spills 408 bytes of stores, in the FP64 logarithm's call.)
template <int G>
constexpr int kWideThreads = G > kTestThreads ? G : kTestThreads;

template <int G, bool DECIDE>
__global__ void __launch_bounds__(kWideThreads<G>) k_pairs_wide(const ProblemDev* __restrict__ probs,
                                                             const int32_t* __restrict__ vtx_prob,
                                                             const int32_t* __restrict__ vtx_first, int total_vertices,
                                                             int max_n, int emit, int sym, int32_t* G_out, long long ldg,
                                                             CritTableDev crit, double alpha, DepthCounters* ctr, int stat,
                                                             int df_mode)
{
    constexpr int NG = kWideThreads<G> / G, kValues = G == 32 ? 32 : 256;
    __shared__ int s_i[NG][kValues], s_j[NG][kValues];      // single counts of i and j
    __shared__ int s_x0[NG][kValues], s_0y[NG][kValues];    // the cells (x, 0) and (0, y); (0, 0) in s_x0
    __shared__ double red[32];
    if (DECIDE && !ctr->active) return;
    const int g = Grp<G>::gid(), r = Grp<G>::rank(), lane = threadIdx.x & 31;
    int *ci = s_i[g], *cj = s_j[g], *x0 = s_x0[g], *y0 = s_0y[g];
    // entry 0 of counts whose values 1 .. m - 1 are set: `all` minus their sum (the group's first warp)
    auto rest_of = [&](int* v, int m, int all) {
        int s = 0;
        for (int k = 1 + lane; k < m; k += 32) s += v[k];
        s = __reduce_add_sync(0xffffffffu, s);
        if (lane == 0) v[0] = all - s;
    };
    unsigned long long removed = 0, tests = 0, samples = 0;   // thread 0 of the group
    const long long tasks = (long long)total_vertices * max_n;
    for (long long t = (long long)blockIdx.x * NG + g; t < tasks; t += (long long)gridDim.x * NG) {
        const int gv = (int)(t / max_n), j = (int)(t - (long long)gv * max_n), p = vtx_prob[gv];
        const ProblemDev& P = probs[p];
        const int i = gv - vtx_first[p], n = P.n;
        if (P.max_arity <= kWideArity || j < i || j >= n) continue;
        const PairGram q(P, i, j);
        const int ri = q.ri, rj = q.rj, N = q.N;
        int32_t* T = emit ? (G_out ? G_out : P.gram) : nullptr;
        const long long ld = G_out ? ldg : P.gram_ld, oi = P.off[i], oj = P.off[j];
        auto put = [&](int x, int y, int v) {
            if (!T) return;
            T[(oi + x) * ld + oj + y] = v;
            if (sym) T[(oj + y) * ld + oi + x] = v;
        };
        for (int x = 1 + r; x < ri; x += G) ci[x] = q.single_i(x);
        for (int y = 1 + r; y < rj; y += G) {
            cj[y] = q.single_j(y);
            y0[y] = 0;
        }
        Grp<G>::sync();
        if (r < 32) {
            rest_of(ci, ri, N);
            rest_of(cj, rj, N);
        }
        Grp<G>::sync();
        if (j == i) {   // the diagonal block
            if (T)
                for (int c = r; c < ri * ri; c += G) {
                    const int x = c / ri, y = c - x * ri;
                    if (sym || x == y) T[(oi + x) * ld + oi + y] = x == y ? ci[x] : 0;
                }
            if (DECIDE && r == 0) P.adj[(long long)i * n + i] = 0;
            Grp<G>::sync();
            continue;
        }
        for (int x = 1 + (r >> 5); x < ri; x += G / 32) {   // a warp per row
            int row = 0;
            for (int y = 1 + lane; y < rj; y += 32) {
                const int v = q.both(x, y);
                row += v;
                if (v) atomicAdd(&y0[y], v);
                put(x, y, v);
            }
            row = __reduce_add_sync(0xffffffffu, row);
            if (lane == 0) {
                x0[x] = ci[x] - row;
                put(x, 0, ci[x] - row);
            }
        }
        Grp<G>::sync();
        for (int y = 1 + r; y < rj; y += G) {
            y0[y] = cj[y] - y0[y];
            put(0, y, y0[y]);
        }
        if (r < 32) rest_of(x0, ri, cj[0]);
        Grp<G>::sync();
        if (r == 0) put(0, 0, x0[0]);
        if constexpr (DECIDE) {
            double st = 0.0;
            for (int c = r; c < ri * rj; c += G) {
                const int x = c / rj, y = c - x * rj;
                const int v = y == 0 ? x0[x] : x == 0 ? y0[y] : q.both(x, y);
                const long long nx = ci[x], ny = cj[y], a = (long long)v * N, b = nx * ny;
                if (stat == kStatX2) {
                    if (b > 0) {
                        const double d = (double)(a - b);
                        st += d * d / ((double)N * (double)nx * (double)ny);
                    }
                } else if (v > 0) {
                    st += 2.0 * (double)v * log1p((double)(a - b) / (double)b);
                }
            }
            st = grp_sum<G>(st, red);
            if (r < 32) {
                long long df = (long long)(ri - 1) * (rj - 1);
                if (df_mode) {
                    int ax = 0, ay = 0;
                    for (int x = lane; x < ri; x += 32) ax += ci[x] > 0;
                    for (int y = lane; y < rj; y += 32) ay += cj[y] > 0;
                    ax = __reduce_add_sync(0xffffffffu, ax);
                    ay = __reduce_add_sync(0xffffffffu, ay);
                    df = (long long)(ax - 1) * (ay - 1);
                }
                if (lane == 0) {
                    const bool dec = df <= 0 || st < crit_get(crit, df, alpha, &ctr->status);   // df 0: p = 1 > alpha
                    P.adj[(long long)i * n + j] = P.adj[(long long)j * n + i] = (uint8_t)!dec;
                    P.sep_len[(long long)i * n + j] = dec ? 0 : -1;
                    P.sep_off[(long long)i * n + j] = 0;
                    removed += dec;
                    tests += 1;
                    samples += (unsigned long long)N;
                }
            }
        }
        Grp<G>::sync();
    }
    if constexpr (DECIDE) {
        if (r == 0 && tests) {   // one test per pair
            atomicAdd(&ctr->removed, removed);
            atomicAdd(&ctr->tests, tests);
            atomicAdd(&ctr->tests_oracle, tests);
            atomicAdd(&ctr->test_samples, samples);
        }
        __syncthreads();
        if (threadIdx.x == 0)
            if (DepthRecord* rec = depth_rec(ctr, ctr->d)) atomicMax(&rec->t_tests_end, gtime());
    }
}

// Zero the pad rows M..Mp of every problem's one-hot matrix (one CTA per
// problem); rows below M are rewritten by k_onehot on every call.
__global__ void k_zero_pad(const ProblemDev* __restrict__ probs)
{
    const ProblemDev& P = probs[blockIdx.x];
    const long long M = (long long)P.roff[P.n - 1] + P.ar[P.n - 1] - 1;
    uint4* E = reinterpret_cast<uint4*>(P.onehot + M * P.onehot_ld);
    const long long n = (P.rgram_ld - M) * P.onehot_ld / 16;
    for (long long q = threadIdx.x; q < n; q += blockDim.x) E[q] = make_uint4(0, 0, 0, 0);
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

}  // namespace

size_t gram_smem_bytes() { return kGramSmem; }

int gram_rows_padded(int M) { return (M + kTile - 1) / kTile * kTile; }

long long gram_samples_padded(long long N) { return (N + kKSlice - 1) / kKSlice * kKSlice; }

cudaError_t launch_onehot(const ProblemDev* probs, const int32_t* vtx_prob, const int32_t* vtx_first,
                          int total_vertices, const DepthCounters* ctr, cudaStream_t st)
{
    k_onehot<<<total_vertices, 256, 0, st>>>(probs, vtx_prob, vtx_first, total_vertices, ctr);
    return cudaGetLastError();
}

cudaError_t launch_zero_pad(const ProblemDev* probs, int nprob, cudaStream_t st)
{
    k_zero_pad<<<nprob, 256, 0, st>>>(probs);
    return cudaGetLastError();
}

cudaError_t encode_onehot_map(void* map, const uint8_t* E, int Mp, long long K)
{
    auto encode = encode_fn();
    if (!encode) return cudaErrorNotSupported;
    cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)Mp};
    cuuint64_t strides[1] = {(cuuint64_t)K};
    cuuint32_t box[2] = {(cuuint32_t)kKSlice, (cuuint32_t)kTile};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = encode(reinterpret_cast<CUtensorMap*>(map), CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<uint8_t*>(E),
                        dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

size_t tensor_map_bytes() { return sizeof(CUtensorMap); }

// Stages (128 samples each) per work unit for problems of tiles[p] output tiles
// over stages[p] stages: the count up to the exact accumulation's for which the
// CTA with the most work ends first.  Its rounds over the units cost a unit's
// stages, or the epilogue of the unit before where that takes longer, and one
// epilogue stays at the end.  An epilogue is 32,768 atomic additions, and with every
// SM busy the chip takes some 370 per ns: 13.5 us, 45 stages (thousand variables at
// 200,000 samples with units of 8 stages: 2,140 us instead of 730).  300 variables at
// 20,011 samples, 9 tiles of 157 stages: 144 units of 10 stages in one round, 95 us
// with the transfers, where powers of two had given 180 of 8 in two, 109 us; units of
// 32 stages take 104 us.
int gram_unit_slices(const long long* tiles, const long long* stages, int k, int num_sms)
{
    long long best = -1;
    int unit = kSlicesPerChunk;
    for (int s = kSlicesPerChunk; s >= 8; --s) {
        long long units = 0, whole = 0;
        for (int p = 0; p < k; ++p) {
            units += tiles[p] * ((stages[p] + s - 1) / s);
            whole += tiles[p] * (stages[p] / s);
        }
        const long long before = (units + num_sms - 1) / num_sms - 1;   // rounds before the last
        const long long last = k == 1 && before * num_sms >= whole ? stages[0] % s : s;
        const long long cost = before * std::max(s, kEpilogueStages) + last + kEpilogueStages;
        if (best < 0 || cost < best) {
            best = cost;
            unit = s;
        }
    }
    return unit;
}

int gram_chunks(long long K, int unit_slices) { return (int)((K / kKSlice + unit_slices - 1) / unit_slices); }

// Gram of every problem's one-hot matrix over the given work units; each
// problem's Gram must be zero.  maps: device array of tensor maps (one per
// problem, 64-byte aligned).
cudaError_t launch_gram(const void* maps, const int4* units, int n_units, int unit_slices, const ProblemDev* probs,
                        int num_sms, unsigned* status, int wait_limit, cudaStream_t st)
{
    GramArgs g;
    g.maps = reinterpret_cast<const CUtensorMap*>(maps);
    g.units = units;
    g.probs = probs;
    g.n_units = n_units;
    g.unit_slices = unit_slices;
    g.status = status;
    g.limit = wait_limit < 0 ? 0u : wait_limit == 0 ? kSpinLimit : (unsigned)wait_limit;
    cudaError_t e = cudaFuncSetAttribute(k_gram, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGramSmem);
    if (e != cudaSuccess) return e;
    const int grid = n_units < num_sms ? n_units : num_sms;
    if (grid <= 0) return cudaSuccess;
    k_gram<<<grid, kGramThreads, kGramSmem, st>>>(g);
    return cudaGetLastError();
}

cudaError_t launch_pairs_gram(const ProblemDev* probs, const int32_t* vtx_prob, const int32_t* vtx_first,
                              int total_vertices, int max_n, const PairsGramArgs& a, int num_sms, cudaStream_t st)
{
    const int blocks_n = (max_n + 31) / 32;
    const long long warps = (long long)total_vertices * blocks_n;
    const int grid = (int)std::max<long long>(1, std::min<long long>((warps + 7) / 8, (long long)num_sms * 8));
    auto kern = a.ctr ? k_pairs_gram<true> : k_pairs_gram<false>;
    kern<<<grid, 256, 0, st>>>(probs, vtx_prob, vtx_first, total_vertices, blocks_n, a.emit, a.sym, a.out, a.ldo,
                               a.total_pairs, a.crit, a.alpha, a.ctr, a.stat, a.df_mode);
    if (a.max_arity > kWideArity) {
        const long long tasks = (long long)total_vertices * max_n;
        auto launch = [&](auto wide, int per_cta, int threads) {
            wide<<<(int)std::min<long long>((tasks + per_cta - 1) / per_cta, (long long)num_sms * (2048 / threads)), threads, 0, st>>>(
                probs, vtx_prob, vtx_first, total_vertices, max_n, a.emit, a.sym, a.out, a.ldo, a.crit, a.alpha, a.ctr,
                a.stat, a.df_mode);
        };
        if (a.max_arity <= 32) launch(a.ctr ? k_pairs_wide<32, true> : k_pairs_wide<32, false>, kTestThreads / 32, kTestThreads);
        else if (a.max_arity <= 64) launch(a.ctr ? k_pairs_wide<kTestThreads, true> : k_pairs_wide<kTestThreads, false>, 1, kTestThreads);
        else launch(a.ctr ? k_pairs_wide<kBigThreads, true> : k_pairs_wide<kBigThreads, false>, 1, kBigThreads);
    }
    return cudaGetLastError();
}

}  // namespace fbn
