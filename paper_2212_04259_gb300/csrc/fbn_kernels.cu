// fbn_kernels.cu -- per-depth kernels of the PC-stable skeleton (Algorithm 1)
// and their host launchers, for sm_103a.  The work-pool kernels live in
// fbn_pool_small.cu, fbn_pool_big.cu, fbn_pool_mid.cu, fbn_plain.cu (device code in
// fbn_pool.cuh) and fbn_pool_marg.cu; the explicit-test kernel in fbn_ci.cu.
//
// Depth pipeline (every kernel runs over all problems of a batch at once):
//   k_snapshot   a(v) for every vertex: adjacency row -> ascending neighbour list
//   k_edges      edges i<j with at least one test, with their rank space
//                |X-side| + |Y-side|, split into a warp class (tables that fit
//                a warp's share of shared memory) and a CTA class
//   k_scan / k_place
//                order each class by chunk count (counted by k_edges), so that
//                pass k of the work pool is a prefix of that order
//   k_pool_*     persistent CI-level work pool (Section IV-B): each group (a
//                warp or a CTA) claims work items -- one chunk of gs
//                consecutive conditioning sets of one edge -- from one atomic
//                counter; items are laid out pass by pass, so every live edge
//                gets its k-th chunk before any edge gets its (k+1)-th; chunks
//                above an edge's lowest accepting rank are skipped
//   k_pool_marg  the pool of depth 1 from one-hot planes (fbn_pool_marg.cuh)
//   k_plain      edge-level form (Section IV-A): one CTA per edge, sequential
//                conditioning sets with early exit
//   k_apply      end-of-depth removal over the snapshot; the separating set is
//                the conditioning set of the lowest accepting rank
//   k_depth_end  records the depth, decides whether Algorithm 1 goes on and
//                clears the per-depth counters for the next depth
//   k_gate       the loop's condition after the next depth's edge list
// Every kernel reads the depth and the sizes from the device counters, so one
// captured sequence serves every depth (the body of the depth loop's while
// node); a kernel that runs after the loop ended finds active == 0 and does
// nothing.  Small calls run the same phases inside one kernel (fbn_loop.cu).
#include <cstdint>
#include <cuda_runtime.h>

#include "fbn_graph.cuh"
#include "fbn_launch.h"

namespace fbn {

// Launches of the depth kernels go through launch_pdl; set_pdl(false)
// launches them without the attribute, on this thread (a capture's retry).
static thread_local bool g_pdl = true;

// The work-pool kernels, each defined in its own translation unit.
__global__ void k_pool_small(PoolArgs a);
__global__ void k_pool_marg(PoolArgs a);
__global__ void k_pairs_popc(const ProblemDev* probs, const int32_t* vtx_prob, const int32_t* vtx_first,
                             int total_vertices, int max_n, const uint8_t* owned, PoolArgs a);
__global__ void k_pool_big(PoolArgs a);
__global__ void k_pool_mid(PoolArgs a);
__global__ void k_plain(PoolArgs a);

// --------------------------------------------------------------------------
__global__ void k_snapshot(const ProblemDev* __restrict__ probs, const int32_t* __restrict__ vtx_prob,
                           const int32_t* __restrict__ vtx_first, int total_vertices, DepthCounters* ctr)
{
    pdl_enter();
    const int g = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (g < total_vertices && ctr->active) snapshot_vertex(probs, vtx_prob, vtx_first, g, ctr, depth_rec(ctr, ctr->d));
}

__global__ void k_edges(const ProblemDev* __restrict__ probs, const int32_t* __restrict__ vtx_prob,
                        const int32_t* __restrict__ vtx_first, int total_vertices, int gs_forced, long long gs_edges,
                        const long long* __restrict__ binom, int brows, long long warp_cells_cap, long long marg_warps,
                        const uint8_t* __restrict__ owned, EdgeWork* __restrict__ edges,
                        unsigned long long* __restrict__ min_accept, long long edge_cap, DepthCounters* ctr,
                        unsigned long long* __restrict__ hist)
{
    pdl_enter();
    const int g = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (g < total_vertices && ctr->active)
        edges_vertex(probs, vtx_prob, vtx_first, g, gs_forced, gs_edges, binom, brows, warp_cells_cap, marg_warps,
                     owned, edges, min_accept, edge_cap, ctr, hist);
}

// One CTA per class.
__global__ void k_scan(ScanClass c0, ScanClass c1, DepthCounters* ctr, double mean_n, int forced_group,
                       long long split_stride, int allow_split, int marg, int need_marg)
{
    pdl_enter();
    if (!ctr->active) return;
    scan_class(blockIdx.x == 0 ? c0 : c1, blockIdx.x, ctr, mean_n, forced_group, split_stride, allow_split, marg,
               need_marg);
}

__global__ void k_place(const ProblemDev* __restrict__ probs, const EdgeWork* __restrict__ edges, long long edge_cap,
                        int nclass, const DepthCounters* ctr, const unsigned long long* __restrict__ alive0,
                        unsigned long long* __restrict__ cursor0, const unsigned long long* __restrict__ alive1,
                        unsigned long long* __restrict__ cursor1, int32_t* __restrict__ sorted)
{
    pdl_enter();
    if (!ctr->active) return;
    place_edges(probs, edges, edge_cap, nclass, ctr, alive0, cursor0, alive1, cursor1, sorted,
                (long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x);
}

__global__ void k_apply(const ProblemDev* __restrict__ probs, const EdgeWork* __restrict__ edges,
                        const unsigned long long* __restrict__ min_accept, long long edge_cap,
                        const long long* __restrict__ binom, int32_t* __restrict__ sep_pool, long long sep_cap,
                        DepthCounters* ctr)
{
    pdl_enter();
    if (!ctr->active) return;
    apply_edges(probs, edges, min_accept, edge_cap, binom, sep_pool, sep_cap, ctr,
                (long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x);
}

__global__ void k_depth_end(DepthCounters* ctr, DepthRecord* rec, int max_depth, unsigned long long* hist,
                            unsigned long long* cursor)
{
    pdl_enter();
    if (!ctr->active) return;
    depth_end(ctr, rec, max_depth, hist, cursor, true);
}

// Sharded skeletons (several processes test shares of one problem's edges):
// the depth's removals of this process's edges as (i, j, lowest accepting
// rank) records, without applying them; the oracle-equivalent test counts as
// k_apply keeps them.
__global__ void k_export_removed(const ProblemDev* __restrict__ probs, const EdgeWork* __restrict__ edges,
                                 const unsigned long long* __restrict__ min_accept, long long edge_cap,
                                 DepthCounters* ctr, long long* __restrict__ out, unsigned long long* __restrict__ count)
{
    pdl_enter();
    if (!ctr->active) return;
    const long long n0 = (long long)ctr->n_edges[0], n1 = (long long)ctr->n_edges[1];
    unsigned long long my_tests = 0, my_samples = 0;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n0 + n1;
         k += (long long)gridDim.x * blockDim.x) {
        const long long e = k < n0 ? k : edge_cap - n1 + (k - n0);
        const EdgeWork w = edges[e];
        const unsigned long long ma = min_accept[e];
        const bool rm = ma < (unsigned long long)w.total;
        const unsigned long long t = rm ? ma + 1 : (unsigned long long)w.total;
        my_tests += t;
        my_samples += t * (unsigned long long)probs[w.prob].N;
        if (rm) {
            const unsigned long long pos = atomicAdd(count, 1ULL);   // < edges of the depth <= edge_cap
            out[3 * pos] = w.i;
            out[3 * pos + 1] = w.j;
            out[3 * pos + 2] = (long long)ma;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        my_tests += __shfl_xor_sync(0xffffffffu, my_tests, o);
        my_samples += __shfl_xor_sync(0xffffffffu, my_samples, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (my_tests) atomicAdd(&ctr->tests_oracle, my_tests);
        if (my_samples) atomicAdd(&ctr->test_samples, my_samples);
    }
}

// Sharded skeletons: remove every process's records of the depth from the
// snapshot (identical on every process) and keep the separating set of each:
// the conditioning set of its rank in the order of k_edges (X-side subsets of
// a(i)\{j} first, then Y-side subsets of a(j)\{i}, each lexicographic).
// Records were validated on the host (i < j < n, adjacent, rank within the
// edge's rank space).
__global__ void k_apply_list(const ProblemDev* __restrict__ probs, const long long* __restrict__ list, long long n_list,
                             const long long* __restrict__ binom, int brows, int32_t* __restrict__ sep_pool,
                             long long sep_cap, DepthCounters* ctr)
{
    pdl_enter();
    if (!ctr->active) return;
    const int d = ctr->d;
    const ProblemDev P = probs[0];
    const long long n = P.n;
    unsigned long long my_removed = 0;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n_list;
         t += (long long)gridDim.x * blockDim.x) {
        const int i = (int)list[3 * t], j = (int)list[3 * t + 1];
        const long long ma = list[3 * t + 2];
        my_removed += 1;
        P.adj[i * n + j] = 0;
        P.adj[j * n + i] = 0;
        long long off = 0;
        if (d > 0) {
            const long long cnt_i = binom_sat(binom, brows, P.deg[i] - 1, d);
            const bool xside = ma < cnt_i;
            const int a = xside ? i : j;
            const int posb = xside ? P.npos[(long long)i * n + j] : P.npos[(long long)j * n + i];
            const long long lr = xside ? ma : ma - cnt_i;
            off = (long long)atomicAdd(&ctr->sep_used, (unsigned long long)d);
            if (off + d > sep_cap) {
                atomicOr(&ctr->status, kStatusSepPool);
                off = 0;
            } else {
                int pos[kMaxD];
                unrank_lex(lr, P.deg[a] - 1, d, binom, pos);
                const int32_t* nb = P.nbr + (long long)a * n;
                for (int q = 0; q < d; ++q) sep_pool[off + q] = nb[pos[q] < posb ? pos[q] : pos[q] + 1];
            }
        }
        P.sep_len[i * n + j] = d;
        P.sep_off[i * n + j] = off;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) my_removed += __shfl_xor_sync(0xffffffffu, my_removed, o);
    if ((threadIdx.x & 31) == 0 && my_removed) atomicAdd(&ctr->removed, my_removed);
}

// The next depth of a sharded skeleton runs whatever this process's share
// held: the host decides when Algorithm 1 stops.
__global__ void k_shard_continue(DepthCounters* ctr)
{
    pdl_enter();
    if (ctr->status == 0) ctr->active = 1;
}

// Condition of the depth loop's graph (one thread), after the edge list of
// the next depth: go on while Algorithm 1 continues and the depth has an edge
// to test (no edge with a side of at least d candidates: the loop ends).
__global__ void k_gate(DepthCounters* ctr, cudaGraphConditionalHandle loop)
{
    pdl_enter();
    const bool go = ctr->active && ctr->n_edges[0] + ctr->n_edges[1] > 0;
    if (!go) ctr->active = 0;
    cudaGraphSetConditional(loop, go ? 1u : 0u);
}

// --------------------------------------------------------------------------
// host launchers

// Launch with programmatic stream serialisation (see pdl_enter).
template <typename... KArgs, typename... Args>
static void launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g_pdl ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

void launch_snapshot(const ProblemDev* probs, const int32_t* vtx_prob, const int32_t* vtx_first,
                     int total_vertices, DepthCounters* ctr, cudaStream_t st)
{
    const int warps = 8;
    launch_pdl(k_snapshot, dim3((total_vertices + warps - 1) / warps), dim3(warps * 32), 0, st, probs, vtx_prob,
               vtx_first, total_vertices, ctr);
}

void launch_edges(const ProblemDev* probs, const int32_t* vtx_prob, const int32_t* vtx_first,
                  int total_vertices, int gs_forced, long long gs_edges, const long long* binom, int brows,
                  long long warp_cells_cap, long long marg_warps, const uint8_t* owned,
                  EdgeWork* edges, unsigned long long* min_accept, long long edge_cap, DepthCounters* ctr,
                  unsigned long long* hist, cudaStream_t st)
{
    const int warps = 8;
    launch_pdl(k_edges, dim3((total_vertices + warps - 1) / warps), dim3(warps * 32), 0, st, probs, vtx_prob,
               vtx_first, total_vertices, gs_forced, gs_edges, binom, brows, warp_cells_cap, marg_warps, owned, edges,
               min_accept, edge_cap, ctr, hist);
}

void launch_order(const ProblemDev* probs, const EdgeWork* edges, long long edge_cap, int nclass, DepthCounters* ctr,
                  const ScanClass* sc, unsigned long long* cursor0, unsigned long long* cursor1, int32_t* sorted,
                  double mean_n, int forced_group, long long split_stride, int allow_split, int marg, int need_marg,
                  int grid, cudaStream_t st)
{
    launch_pdl(k_scan, dim3(nclass), dim3(256), 0, st, sc[0], sc[nclass > 1 ? 1 : 0], ctr, mean_n, forced_group,
               split_stride, allow_split, marg, need_marg);
    launch_pdl(k_place, dim3(grid), dim3(256), 0, st, probs, edges, edge_cap, nclass, ctr, (const unsigned long long*)sc[0].alive,
               cursor0, (const unsigned long long*)sc[nclass > 1 ? 1 : 0].alive, cursor1, sorted);
}

void launch_pool(const PoolArgs& a, int cls, int grid, size_t smem_bytes, cudaStream_t st)
{
    if (cls == kClassWarp) launch_pdl(k_pool_small, dim3(grid), dim3(kTestThreads), smem_bytes, st, a);
    else launch_pdl(k_pool_big, dim3(grid), dim3(kBigThreads), smem_bytes, st, a);
}

void launch_pool_mid(const PoolArgs& a, int grid, size_t smem_bytes, cudaStream_t st)
{
    launch_pdl(k_pool_mid, dim3(grid), dim3(kTestThreads), smem_bytes, st, a);
}

void launch_pool_marg(const PoolArgs& a, int grid, cudaStream_t st)
{
    launch_pdl(k_pool_marg, dim3(grid), dim3(kMargThreads), 0, st, a);
}

void launch_pairs_popc(const ProblemDev* probs, const int32_t* vtx_prob, const int32_t* vtx_first, int total_vertices,
                       int max_n, const uint8_t* owned, const PoolArgs& a, int grid, cudaStream_t st)
{
    launch_pdl(k_pairs_popc, dim3(grid), dim3(kTestThreads), 0, st, probs, vtx_prob, vtx_first, total_vertices, max_n,
               owned, a);
}

void launch_plain(const PoolArgs& a, int grid, size_t smem_bytes, cudaStream_t st)
{
    launch_pdl(k_plain, dim3(grid), dim3(kTestThreads), smem_bytes, st, a);
}

void launch_apply(const ProblemDev* probs, const EdgeWork* edges, const unsigned long long* min_accept,
                  long long edge_cap, const long long* binom, int32_t* sep_pool, long long sep_cap,
                  DepthCounters* ctr, int grid, cudaStream_t st)
{
    launch_pdl(k_apply, dim3(grid), dim3(256), 0, st, probs, edges, min_accept, edge_cap, binom, sep_pool, sep_cap,
               ctr);
}

void launch_shard_export(const ProblemDev* probs, const EdgeWork* edges, const unsigned long long* min_accept,
                         long long edge_cap, DepthCounters* ctr, long long* out, unsigned long long* count, int grid,
                         cudaStream_t st)
{
    launch_pdl(k_export_removed, dim3(grid), dim3(256), 0, st, probs, edges, min_accept, edge_cap, ctr, out, count);
}

void launch_shard_apply(const ProblemDev* probs, const long long* list, long long n_list, const long long* binom,
                        int brows, int32_t* sep_pool, long long sep_cap, DepthCounters* ctr, int grid, cudaStream_t st)
{
    launch_pdl(k_apply_list, dim3(grid), dim3(256), 0, st, probs, list, n_list, binom, brows, sep_pool, sep_cap, ctr);
}

void launch_shard_continue(DepthCounters* ctr, cudaStream_t st)
{
    launch_pdl(k_shard_continue, dim3(1), dim3(1), 0, st, ctr);
}

void launch_depth_end(DepthCounters* ctr, DepthRecord* rec, int max_depth, unsigned long long* hist,
                      unsigned long long* cursor, cudaStream_t st)
{
    launch_pdl(k_depth_end, dim3(1), dim3(256), 0, st, ctr, rec, max_depth, hist, cursor);
}

void launch_gate(DepthCounters* ctr, cudaGraphConditionalHandle loop, cudaStream_t st)
{
    launch_pdl(k_gate, dim3(1), dim3(1), 0, st, ctr, loop);
}

void set_pdl(bool on)
{
    g_pdl = on;
}

cudaError_t set_kernel_smem(size_t small_smem, size_t big_smem, size_t cta_smem)
{
    cudaError_t e;
    const int b = (int)cta_smem;
    if ((e = cudaFuncSetAttribute(k_pool_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)small_smem))) return e;
    if ((e = cudaFuncSetAttribute(k_pool_big, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)big_smem))) return e;
    if ((e = cudaFuncSetAttribute(k_pool_mid, cudaFuncAttributeMaxDynamicSharedMemorySize, b))) return e;
    if ((e = cudaFuncSetAttribute(k_plain, cudaFuncAttributeMaxDynamicSharedMemorySize, b))) return e;
    return cudaSuccess;
}

int pool_blocks_per_sm(int cls, size_t smem_bytes)
{
    int nb = 0;
    if (cls == kClassMarg)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_pool_marg, kMargThreads, smem_bytes);
    else if (cls == kClassWarp)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_pool_small, kTestThreads, smem_bytes);
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_pool_big, kBigThreads, smem_bytes);
    return nb;
}

}  // namespace fbn
