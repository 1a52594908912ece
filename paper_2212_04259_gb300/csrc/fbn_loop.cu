// fbn_loop.cu -- the whole skeleton of a small problem as one persistent kernel.
//
// What bounds small problems is not their tests but the way from one depth to
// the next: nine kernels and a while node a depth, 37-41 us of which the tests
// were 5 to 10, and a dozen launches and memsets before the loop.  Here one
// cooperative launch runs every depth; its CTAs meet at a barrier between the
// phases, and short serial work (ordering, the end of a depth) is done by the
// CTA that arrives last, before it opens the barrier:
//   init | snapshot (+ end of the depth before) | edge list (+ ordering) | tests
//   | removal
// and at the end the results, separating sets included, go straight to pinned
// host memory.
// The phases are those of the per-depth kernels (fbn_graph.cuh, fbn_pool.cuh,
// fbn_pool_marg.cuh), so the results are too.  Larger problems keep the
// kernels: their phases fill the chip, and the fixed cost per depth no longer
// shows.  So does a depth with a table over the loop's shared memory: the loop
// ends before that depth's removal and the graph goes on there, whose big-table
// pools have 100 to 200 KB (20 variables of 12 values x 50,000 samples to depth 2,
// 20,736 cells: 48 ms with these tables in global memory, 9.0 handed over; 14
// variables of 7 values to depth 3, 16,807 cells: 33 and 5.5 ms).
#include "fbn_graph.cuh"
#include "fbn_loop.h"
#include "fbn_pool_marg.cuh"
#include "fbn_turn.cuh"

namespace fbn {
namespace {

constexpr long long kPlaceSerial = 2048;   // edges the last CTA of the edge list orders by itself

constexpr unsigned kGaveUp = 1u << 31;   // bar[0]: the phase will not open

__device__ __forceinline__ unsigned phases_open(const unsigned* bar)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&bar[1]) : "memory");
    return v;
}

// A CTA that has waited too long marks the phase as given up, unless it is open
// or about to be; true when it is given up.  The mark goes on a count that still
// lacks a CTA, and the CTA that completes a marked count does not open the phase:
// so every CTA passes a barrier, or none.  (A count read or marked may belong to
// the next phase when this one has opened meanwhile; the open word, read after a
// fence, tells, and the next phase is then given up by all.)
__device__ __noinline__ bool give_up(unsigned* bar, unsigned gen)
{
    unsigned w = *((volatile unsigned*)&bar[0]);
    for (;;) {
        __threadfence();
        if (phases_open(bar) == gen + 1) return false;
        if (w & kGaveUp) return true;
        if (w == 0 || w == gridDim.x) return false;   // everyone is here: the last one is opening it
        const unsigned old = atomicCAS(&bar[0], w, w | kGaveUp);
        if (old == w) {
            __threadfence();
            return phases_open(bar) != gen + 1;
        }
        w = old;
    }
}

// All CTAs of the (cooperative) grid; the one that arrives last runs `last`
// first.  The wait is bounded: after a.spin_limit polls during which no CTA claimed
// an item or finished a test within one, the waiting CTA gives the phase up; every
// CTA then leaves (false), and the host runs the call as a graph.
template <class Last>
__device__ __forceinline__ bool loop_barrier(const LoopArgs& a, unsigned& gen, Last last)
{
    __shared__ int s_role;   // 1: the last to arrive; 0: waited; -1: gave up
    unsigned* bar = a.bar;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned before = atomicAdd(&bar[0], 1u);
        s_role = before == gridDim.x - 1 ? 1 : before & kGaveUp ? -1 : 0;
    }
    __syncthreads();
    if (s_role == 1) {
        __threadfence();
        last();
        __syncthreads();
        if (threadIdx.x == 0) {
            bar[0] = 0;   // nobody arrives again before the phase is open
            __threadfence();
            asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(&bar[1]), "r"(gen + 1) : "memory");
        }
    } else if (s_role == 0 && threadIdx.x == 0) {
        unsigned long long seen = ~0ULL;
        unsigned it = 0;
        while (phases_open(bar) != gen + 1) {
            if (it++ < a.spin_limit) continue;
            const volatile DepthCounters* c = a.ctr;
            const unsigned long long now = c->next_item[0] + c->next_item[1] + c->beat;   // items claimed, tests within them
            if ((now == seen || a.spin_limit == 0) && give_up(bar, gen)) {
                s_role = -1;
                break;
            }
            seen = now;
            it = 0;
        }
        __threadfence();
    }
    __syncthreads();
    ++gen;
    if (s_role < 0 && threadIdx.x == 0) *((volatile unsigned*)a.left) = kLoopGaveUp;
    return s_role >= 0;
}

// The results to pinned host memory (one problem), after the last depth.
__device__ __forceinline__ void loop_results(const LoopArgs& a, unsigned& gen, int warp0, int warps, long long t0,
                                             long long threads)
{
    const ProblemDev& P = a.probs[0];
    const int n = P.n, lane = threadIdx.x & 31;
    const unsigned status = a.ctr->status;
    if (a.h_adj) {   // whole 16-byte words: both buffers are padded
        const uint4* src = reinterpret_cast<const uint4*>(P.adj);
        uint4* dst = reinterpret_cast<uint4*>(a.h_adj);
        for (long long k = t0; k < ((long long)n * n + 15) / 16; k += threads) dst[k] = src[k];
    }
    if (status == 0) {
        for (int i = warp0; i < n; i += warps) {   // pairs and members of row i
            int pairs = 0, members = 0;
            for (int j = i + 1 + lane; j < n; j += 32) {
                const int L = P.sep_len[(long long)i * n + j];
                pairs += L >= 0;
                members += L > 0 ? L : 0;
            }
            pairs = __reduce_add_sync(0xffffffffu, pairs);
            members = __reduce_add_sync(0xffffffffu, members);
            if (lane == 0) {
                a.sep_cnt[i] = pairs;
                a.sep_cnt[n + i] = members;
            }
        }
    }
    // every depth's counters are final here
    if (blockIdx.x == 0) {
        const unsigned* src = reinterpret_cast<const unsigned*>(a.ctr);
        unsigned* dst = reinterpret_cast<unsigned*>(a.h_ctr);
        for (int k = threadIdx.x; k < (int)(sizeof(DepthCounters) / 4); k += kTestThreads) dst[k] = src[k];
        src = reinterpret_cast<const unsigned*>(a.rec);
        dst = reinterpret_cast<unsigned*>(a.h_rec);
        for (int k = threadIdx.x; k < (int)(kMaxDepthRecords * sizeof(DepthRecord) / 4); k += kTestThreads) dst[k] = src[k];
    }
    if (status != 0) return;   // the same for every CTA: nothing changes it any more
    if (!loop_barrier(a, gen, [] {})) return;
    for (int i = warp0; i < n; i += warps) {
        int p = 0, m = 0;   // pairs and members of the rows before i
        for (int r = lane; r < i; r += 32) {
            p += (int)a.sep_cnt[r];
            m += (int)a.sep_cnt[n + r];
        }
        p = __reduce_add_sync(0xffffffffu, p);
        m = __reduce_add_sync(0xffffffffu, m);
        for (int j0 = i + 1; j0 < n; j0 += 32) {
            const int j = j0 + lane;
            const int L = j < n ? P.sep_len[(long long)i * n + j] : -1;
            const unsigned take = __ballot_sync(0xffffffffu, L >= 0);
            int inc = L > 0 ? L : 0;   // inclusive scan of the lengths
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            if (L >= 0) {
                const int k = p + __popc(take & ((1u << lane) - 1u));
                const int mo = m + inc - L;
                a.h_pairs[2 * k] = i;
                a.h_pairs[2 * k + 1] = j;
                a.h_offs[k] = mo;
                const int32_t* src = a.sep_pool + P.sep_off[(long long)i * n + j];
                for (int q = 0; q < L; ++q) a.h_members[mo + q] = src[q];
            }
            p += __popc(take);
            m += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (i == n - 1 && lane == 0) {
            a.h_tot[0] = p;
            a.h_tot[1] = m;
        }
    }
}

__global__ void __launch_bounds__(kTestThreads, 2) k_loop(const __grid_constant__ LoopArgs a)
{
    extern __shared__ __align__(16) int smem[];
    __shared__ PoolShared sh;
    __shared__ TurnShared turn_sh;
    DepthCounters* ctr = a.ctr;
    // phases opened before this launch: none opens before this CTA arrives
    unsigned gen = *((volatile unsigned*)&a.bar[1]);
    const int warp0 = blockIdx.x * (kTestThreads / 32) + (threadIdx.x >> 5), warps = gridDim.x * (kTestThreads / 32);
    const int lane = threadIdx.x & 31;
    const long long t0 = (long long)blockIdx.x * kTestThreads + threadIdx.x, threads = (long long)gridDim.x * kTestThreads;
    auto none = [] {};

    // counters, histograms and the complete graph
    if (blockIdx.x == 0)
        for (int k = threadIdx.x; k < (int)(sizeof(DepthCounters) / 4); k += kTestThreads)
            reinterpret_cast<unsigned*>(ctr)[k] = reinterpret_cast<const unsigned*>(&a.init)[k];
    for (long long k = t0; k < 2 * a.ord_cap; k += threads) a.hist[k] = a.cursor[k] = 0;
    for (long long k = t0; k < (long long)(kMaxDepthRecords * sizeof(DepthRecord) / 8); k += threads)
        reinterpret_cast<unsigned long long*>(a.rec)[k] = 0;
    if (a.bits && blockIdx.x == 0)
        for (int k = threadIdx.x; k < kTurnVertices * (kTurnVertices / 32); k += kTestThreads) {
            const int v = k / (kTurnVertices / 32), w = k - v * (kTurnVertices / 32), n = a.total_vertices;
            const unsigned row = w * 32 + 32 <= n ? ~0u : w * 32 < n ? (1u << (n - w * 32)) - 1u : 0u;
            a.bits[k] = v < n ? (v >> 5 == w ? row & ~(1u << (v & 31)) : row) : 0u;
        }
    for (int g = warp0; g < a.total_vertices; g += warps) {
        const int p = a.vtx_prob[g];
        const ProblemDev& P = a.probs[p];
        const int i = g - a.vtx_first[p], n = P.n;
        for (int j = lane; j < n; j += 32) {
            P.adj[(long long)i * n + j] = (uint8_t)(i != j);
            P.sep_len[(long long)i * n + j] = -1;
            P.sep_off[(long long)i * n + j] = 0;
        }
    }
    if (!loop_barrier(a, gen, none)) return;

    for (int d = 0;; ++d) {
        const bool popc = d == 0 && a.popc0, marg = d == 1 && a.marg1;
        const bool direct = ctr->direct != 0;   // listed by the last CTA of the depth before
        long long big = (long long)ctr->n_edges[kClassCta];   // listed directly, else read below
        if (!direct) {
            // the last CTA ends the depth before, the others list the neighbours
            // (the degree sum, which they add up, was cleared by the phase before)
            if (d > 0 && !a.bits && blockIdx.x == gridDim.x - 1) depth_end(ctr, a.rec, a.max_depth, a.hist, a.cursor, false);
            DepthRecord* begin = d < kMaxDepthRecords ? a.rec + d : nullptr;
            for (int g = warp0; g < a.total_vertices; g += warps)
                snapshot_vertex(a.probs, a.vtx_prob, a.vtx_first, g, ctr, begin);
            if (!loop_barrier(a, gen, none)) return;
            if (!ctr->active) break;   // the same for every CTA
            for (int g = warp0; g < a.total_vertices; g += warps)
                edges_vertex(a.probs, a.vtx_prob, a.vtx_first, g, a.gs_forced, a.gs_edges, a.binom, a.brows,
                             a.warp_cells_cap, marg ? warps : 0, nullptr, a.edges, a.min_accept, a.edge_cap, ctr, a.hist);
            auto place = [&](long long first, long long step) {
                place_edges(a.probs, a.edges, a.edge_cap, marg ? 1 : 2, ctr, a.sc[0].alive, a.cursor, a.sc[1].alive,
                            a.cursor + a.ord_cap, a.sorted, first, step);
            };
            // the last CTA: whether the depth has an edge to test, and the order
            // of its items (none for depth 0 from planes)
            auto order = [&] {
                const long long E0 = (long long)ctr->n_edges[0], E1 = (long long)ctr->n_edges[1], E = E0 + E1;
                __syncthreads();   // every thread has read the counts
                if (threadIdx.x == 0) {
                    ctr->adj_ends = 0;
                    if (E == 0) ctr->active = 0;
                }
                if (E == 0 || popc) return;
                for (int cls = 0; cls < 2; ++cls) {   // class 0, also when empty, notes where the tests begin
                    if (cls && E1 == 0) continue;
                    scan_class(a.sc[cls], cls, ctr, a.mean_n, a.forced_group, a.split_stride, 1, marg, a.need_marg);
                    __syncthreads();
                }
                if (depth_is_heavy(ctr->cost[0] + ctr->cost[1], ctr->d, a.rec)) hand_over(a, ctr);
                else if (E <= kPlaceSerial) place(threadIdx.x, kTestThreads);
            };
            if (!loop_barrier(a, gen, order)) return;
            const long long all = (long long)(ctr->n_edges[0] + ctr->n_edges[1]);
            big = (long long)ctr->n_edges[kClassCta];
            const int active = ctr->active;   // the same for every CTA
            if (active < 0) return;
            if (!active) break;
            if (!popc && all > kPlaceSerial) {
                place(t0, threads);
                if (!loop_barrier(a, gen, none)) return;
            }
        }
        if (popc) {
            pairs_popc_body<true>(a.probs, a.vtx_prob, a.vtx_first, a.total_vertices, a.max_n, nullptr, a.small);
        } else if (marg) {
            marg_body<true>(a.small);
        } else {
            bool small = true;
            if (big > 0) {   // first: a table over the shared memory ends the loop
                __shared__ int s_over;
                pool_body<kTestThreads, true>(a.big, smem, sh);
                __syncthreads();
                if (threadIdx.x == 0) s_over = *((volatile int*)&ctr->hand_over);
                __syncthreads();
                small = !s_over;
            }
            if (small) {
                switch (ctr->gsel) {
                    case 32: pool_body<32, true>(a.small, smem, sh); break;
                    case 64: pool_body<64, true>(a.small, smem, sh); break;
                    case 128: pool_body<128, true>(a.small, smem, sh); break;
                    default: pool_body<kTestThreads, true>(a.small, smem, sh); break;
                }
            }
        }
        tests_done(ctr);
        const auto over = [&] { if (big > 0 && ctr->hand_over) hand_over(a, ctr); };
        const auto next = [&] {
            if (big > 0 && ctr->hand_over) hand_over(a, ctr);
            else if (a.bits) turn(a, turn_sh, direct, warps);
        };
        if (direct) {   // removal, end of depth and the next depth's items
            if (!loop_barrier(a, gen, next)) return;
            if (big > 0 && ctr->active < 0) return;   // set before the barrier: the same for every CTA
        } else {
            if (!loop_barrier(a, gen, over)) return;
            if (big > 0 && ctr->active < 0) return;
            apply_edges(a.probs, a.edges, a.min_accept, a.edge_cap, a.binom, a.sep_pool, a.sep_cap, ctr, t0, threads,
                        a.bits);
            if (!loop_barrier(a, gen, next)) return;
        }
        // turn() set it before the barrier opened.  Without the bit matrix the last
        // CTA may be ending the depth already (depth_end above): every CTA then
        // reads it behind the snapshot's barrier
        if (a.bits) {
            const int active = ctr->active;
            if (active < 0) return;
            if (!active) break;
        }
    }
    if (a.h_ctr) loop_results(a, gen, warp0, warps, t0, threads);
}

}  // namespace

cudaError_t prepare_loop(size_t smem_bytes, int* blocks_per_sm)
{
    cudaError_t e = cudaFuncSetAttribute(k_loop, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_loop, kTestThreads, smem_bytes);
}

cudaError_t launch_loop(const LoopArgs& a, int grid, size_t smem_bytes, cudaStream_t st)
{
    void* args[] = {const_cast<LoopArgs*>(&a)};
    return cudaLaunchCooperativeKernel((const void*)k_loop, dim3(grid), dim3(kTestThreads), args, smem_bytes, st);
}

}  // namespace fbn
