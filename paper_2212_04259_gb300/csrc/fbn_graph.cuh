// fbn_graph.cuh -- the graph side of a depth of Algorithm 1 as device code: the
// adjacency snapshot, the edge list, its ordering for the work pools, the
// removal and the end of the depth.  Used by one kernel each (fbn_kernels.cu)
// and by the persistent loop of small problems (fbn_loop.cu), where the arrays
// change between phases of one kernel: nothing here is read through the
// read-only cache.
#pragma once

#include "fbn_depth.cuh"

namespace fbn {

// a(v) of vertex g (one warp): its adjacency row as an ascending list, and
// every neighbour's place in it.  begin: the depth's record (nullptr: none).
__device__ __forceinline__ void snapshot_vertex(const ProblemDev* probs, const int32_t* vtx_prob,
                                                const int32_t* vtx_first, int g, DepthCounters* ctr,
                                                DepthRecord* begin)
{
    const int lane = threadIdx.x & 31;
    if (g == 0 && lane == 0 && begin) begin->t_begin = gtime();
    const int p = vtx_prob[g];
    const ProblemDev P = probs[p];
    const int v = g - vtx_first[p];
    const uint8_t* row = P.adj + (long long)v * P.n;
    int32_t* out = P.nbr + (long long)v * P.n;
    int count = 0;
    for (int b0 = 0; b0 < P.n; b0 += 256) {   // eight loads in flight per lane
        bool a[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) a[q] = b0 + 32 * q + lane < P.n && row[b0 + 32 * q + lane];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int j = b0 + 32 * q + lane;
            const unsigned m = __ballot_sync(0xffffffffu, a[q]);
            if (a[q]) {
                const int slot = count + __popc(m & ((1u << lane) - 1u));
                out[slot] = j;
                P.npos[(long long)v * P.n + j] = slot;
            }
            count += __popc(m);
        }
    }
    if (lane == 0) {
        P.deg[v] = count;
        atomicAdd((unsigned long long*)&ctr->adj_ends, (unsigned long long)count);
    }
}

// --------------------------------------------------------------------------
__device__ __forceinline__ long long binom_sat(const long long* B, int brows, int n, int k)
{
    if (k < 0 || n < k) return 0;
    if (n >= brows || k >= kBinomCols) return kBinomSat;
    return B[(long long)n * kBinomCols + k];
}

// Depth 1 from one-hot planes: edges per warp from which an item is a whole
// edge (no test beyond the first accepting one, no claim per chunk), and the
// ranks per item from one edge per warp on.  Below, single ranks: the depth is
// then as long as its longest chain of tests.  Measured (depth 1, ms): 4.4 edges
// per warp (1,000 variables) whole 3.70, chunks of 1 / 2 / 4 / 8 ranks 1.73 /
// 1.62 / 1.63 / 1.75; 9 per warp (20 problems) whole 0.73, chunks 0.92 / 0.70 /
// 0.62 / 0.61; 131 per warp (256 problems) whole 5.4.
constexpr long long kWholeEdges = 16;
constexpr int kMargChunk = 4;

// The edges i < j of vertex g = i (one warp) with their rank space, class and
// order key.
__device__ __forceinline__ void edges_vertex(const ProblemDev* probs, const int32_t* vtx_prob,
                                             const int32_t* vtx_first, int g, int gs_forced, long long gs_edges,
                                             const long long* binom, int brows, long long warp_cells_cap,
                                             long long marg_warps, const uint8_t* owned, EdgeWork* edges,
                                             unsigned long long* min_accept, long long edge_cap, DepthCounters* ctr,
                                             unsigned long long* hist)
{
    const int lane = threadIdx.x & 31;
    const int d = ctr->d;
    // ranks per chunk: 1 while the live edges are few against the groups
    // (latency of a single test dominates), 4 when there are many (fewer claims)
    const long long live = (long long)(ctr->adj_ends / 2);
    int gs = gs_forced > 0 ? gs_forced : live >= gs_edges ? 4 : 1;
    // depth 1 from one-hot planes (marg_warps > 0: the warps of its pool): a
    // whole edge per item from kWholeEdges edges per warp
    bool whole = false;
    if (marg_warps > 0 && d == 1 && gs_forced == 0) {
        whole = live >= kWholeEdges * marg_warps;
        gs = live >= marg_warps ? kMargChunk : 1;
    }
    if (g == 0 && lane == 0) {
        ctr->gs = gs;
        ctr->whole = whole;
    }
    const int p = vtx_prob[g];
    const ProblemDev P = probs[p];
    const int i = g - vtx_first[p];
    const int deg_i = P.deg[i];
    const int32_t* nb = P.nbr + (long long)i * P.n;
    unsigned long long mc[2] = {0, 0}, mcell[2] = {0, 0}, mtot[2] = {0, 0};
    for (int t0 = 0; t0 < deg_i; t0 += 32) {
        const int t = t0 + lane;
        int j = -1;
        long long cnt_i = 0, total = 0;
        if (t < deg_i) {
            j = nb[t];
            // owned: the edges this process tests when several share the
            // skeleton (one problem; entry [i][j], i < j); nullptr: every edge
            if (j > i && (owned == nullptr || owned[(long long)i * P.n + j])) {
                if (d == 0) {
                    cnt_i = 1;
                    total = 1;
                } else {
                    cnt_i = binom_sat(binom, brows, deg_i - 1, d);
                    total = cnt_i + binom_sat(binom, brows, P.deg[j] - 1, d);
                }
            }
        }
        unsigned long long cells = 0;
        if (total > 0) {
            // cells bound r_i r_j max_arity^d
            cells = (unsigned long long)P.ar[i] * P.ar[j];
            for (int k = 0; k < d && cells <= (unsigned long long)kMaxCells; ++k)
                cells *= (unsigned long long)P.max_arity;
        }
        const int cls = cells <= (unsigned long long)warp_cells_cap ? kClassWarp : kClassCta;
        {   // histogram of each class's order key: one atomic per distinct bin in the warp
            const long long key = whole ? edge_item_key(total, P.N, P.ar[i], P.ar[j]) : chunk_count(total, gs);
            const long long bin = total > 0 ? (long long)cls * (kMaxPasses + 1) + key : -1;
            const unsigned same = __match_any_sync(0xffffffffu, bin);
            if (bin >= 0 && lane == __ffs(same) - 1) atomicAdd(&hist[bin], (unsigned long long)__popc(same));
        }
        for (int c = 0; c < 2; ++c) {
            const bool take = total > 0 && cls == c;
            const unsigned m = __ballot_sync(0xffffffffu, take);
            unsigned long long base = 0;
            if (lane == 0 && m) base = atomicAdd(&ctr->n_edges[c], (unsigned long long)__popc(m));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (!take) continue;
            const long long k = (long long)base + __popc(m & ((1u << lane) - 1u));
            if (k >= edge_cap) {
                atomicOr(&ctr->status, kStatusEdges);
                continue;
            }
            const long long e = c == kClassWarp ? k : edge_cap - 1 - k;
            const int lo = P.npos[(long long)j * P.n + i];   // position of i in a(j)
            EdgeWork w;
            w.prob = p; w.i = i; w.j = j;
            w.posj = (int16_t)t; w.posi = (int16_t)lo;
            w.cnt_i = cnt_i; w.total = total;
            edges[e] = w;
            min_accept[e] = (unsigned long long)total;
            P.eid[(long long)i * P.n + t] = (int32_t)e;
            P.eid[(long long)j * P.n + lo] = (int32_t)e;
            const unsigned long long ch = (unsigned long long)(whole ? edge_item_key(total, P.N, P.ar[i], P.ar[j]) : chunk_count(total, gs));
            mc[c] = ch > mc[c] ? ch : mc[c];
            mcell[c] = cells > mcell[c] ? cells : mcell[c];
            mtot[c] = (unsigned long long)total > mtot[c] ? (unsigned long long)total : mtot[c];
        }
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long a = __shfl_down_sync(0xffffffffu, mc[c], o);
            const unsigned long long b = __shfl_down_sync(0xffffffffu, mcell[c], o);
            const unsigned long long t = __shfl_down_sync(0xffffffffu, mtot[c], o);
            mc[c] = a > mc[c] ? a : mc[c];
            mcell[c] = b > mcell[c] ? b : mcell[c];
            mtot[c] = t > mtot[c] ? t : mtot[c];
        }
        if (lane == 0) {
            if (mc[c]) atomicMax(&ctr->maxc[c], mc[c]);
            if (mcell[c]) atomicMax(&ctr->max_cells[c], mcell[c]);
            if (mtot[c]) atomicMax(&ctr->max_total[c], mtot[c]);
        }
    }
}

// --------------------------------------------------------------------------
// One CTA: alive[k] = #edges with more than k chunks (k = 0..maxc), base[k] =
// sum_{k' < k} alive[k'] (k = 0..maxc).  base[maxc] is the item count.
// Block-wide scans over contiguous per-thread segments.
__device__ __forceinline__ unsigned long long block_exclusive_scan(unsigned long long v, unsigned long long* sh)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[warp] = x;
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        unsigned long long s = lane < nw ? sh[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < nw) sh[lane] = s;
    }
    __syncthreads();
    const unsigned long long before = warp > 0 ? sh[warp - 1] : 0;
    __syncthreads();
    return before + x - v;
}

// One CTA, one class.  Also picks the group size of the small-table class
// from a cost model of the depth: with W work items and g(G) groups of G
// threads, the pool runs ceil(W / g(G)) rounds of one test each, a test
// costing a fixed latency (claim, setup, merge, decision; ~kTestOverhead
// cycles) plus the counting of N samples over G threads (~kCyclesPerSample
// per sample and thread).  groups[k] = groups of size 32 << k; the caller
// may force a size.
constexpr float kTestOverhead = 10000.0f;
constexpr float kCyclesPerSample = 8.0f;

// One thread, with the depth's maxima and ranks per chunk in ctr: the group
// size of the small-table class and the sample split of class cls for W items;
// returns the estimated cycles of the class's tests.
__device__ __forceinline__ float choose_pool(const ScanClass& sc, int cls, unsigned long long W, DepthCounters* ctr,
                                            double mean_n, int forced_group, long long split_stride, int allow_split,
                                            int need_marg)
{
    const long long g32 = sc.groups[0], g64 = sc.groups[1], g128 = sc.groups[2], g256 = sc.groups[3];
    const long long smem_ints = sc.smem_ints;
    if (cls == 0) {
        const long long groups[4] = {g32, g64, g128, g256};
        int best = kTestThreads;
        float best_t = 3e38f;
        // group sizes whose slice holds the class's largest table (the whole CTA's does)
        const long long mcells = (long long)ctr->max_cells[cls];
        auto fits = [&](int G) { return G >= kTestThreads || mcells <= slice_cells(smem_ints * G / kTestThreads, need_marg); };
        for (int k = 0; k < 4; ++k) {
            const int G = 32 << k;
            if (!fits(G)) continue;
            // one thread: FP32 and no 64-bit division (the FP64 pipe and the
            // division routine took 2 us of a small problem's depth)
            const float rounds = ceilf((float)W / (float)groups[k]);
            const float t = rounds * (kTestOverhead + kCyclesPerSample * (float)mean_n / (float)G);
            if (t < best_t) {
                best_t = t;
                best = G;
            }
        }
        // the caller's choice, the autotuner's for this depth, or the cost model's
        const int tuned = tune_code(ctr->tune, ctr->d) & kTuneGroupMask;
        int G = forced_group ? forced_group : tuned ? tuned : best;
        while (!fits(G)) G *= 2;
        ctr->gsel = G;
    }
    // sample split: few single-rank tests against the groups of the class
    const int G = cls == 0 ? ctr->gsel : kTestThreads;
    const long long groups = cls == 0 ? (G == 32 ? g32 : G == 64 ? g64 : G == 128 ? g128 : g256) : g256;
    const long long slice = smem_ints * G / kTestThreads;
    const long long mcell = (long long)ctr->max_cells[cls];
    long long sp = 1;
    if (allow_split && ctr->gs == 1 && ctr->max_total[cls] <= (unsigned long long)kMaxPasses &&
        (long long)W * 2 <= groups && (long long)W <= kSplitItems && mcell <= split_stride &&
                (mcell * 9) / 4 + 64 <= slice) {
        sp = (int)groups / (int)W;
        const long long by_n = (long long)mean_n / kSplitMinSamples;
        sp = sp < by_n ? sp : by_n;
        sp = sp < kMaxSplit ? sp : kMaxSplit;
        sp = sp > 1 ? sp : 1;
    }
    // the big-table class where the decision needs marginals: CTAs of 256 threads when
    // its tests are more than one round of CTAs of 1,024 and fit their shared memory
    // (a round takes them 44 us against 30, on half as many tests)
    if (cls == 1) ctr->wide = !need_marg || (long long)W <= g256 || mcell > sc.mid_ints;
    ctr->split[cls] = (int)sp;
    ctr->total_items[cls] = W * (unsigned long long)sp;
    // the class's tests in cycles, every rank tested (the ranks of the longest chunk, in FP32: see above)
    const float most = (float)ctr->max_total[cls], ranks = fminf(most, fmaxf((float)ctr->gs, most * (1.0f / (float)kMaxPasses)));
    return ceilf((float)W / (float)groups) * ranks * (kTestOverhead + kCyclesPerSample * (float)mean_n / (float)G);
}

__device__ __forceinline__ void scan_class(const ScanClass& sc, int cls, DepthCounters* ctr, double mean_n,
                                           int forced_group, long long split_stride, int allow_split, int marg,
                                           int need_marg)
{
    __shared__ unsigned long long sh[32];
    if (cls == 0 && threadIdx.x == 0)
        if (DepthRecord* r = depth_rec(ctr, ctr->d)) r->t_tests = gtime();
    const unsigned long long* hist = sc.hist;
    unsigned long long* alive = sc.alive;
    unsigned long long* base = sc.base;
    const long long maxc = (long long)ctr->maxc[cls];
    if (ctr->n_edges[cls] == 0) return;
    const int T = blockDim.x;
    const long long len = maxc + 1;
    const long long seg = (len + T - 1) / T;
    // alive[c] = sum_{c' > c} hist[c']: thread t owns the t-th segment counted
    // from the end of the array, so an exclusive scan in thread order sums the
    // segments that lie after this thread's one
    long long lo = len - (long long)(threadIdx.x + 1) * seg, hi = len - (long long)threadIdx.x * seg;
    if (lo < 0) lo = 0;
    if (hi < 0) hi = 0;
    unsigned long long s = 0;
    for (long long c = lo; c < hi; ++c) s += hist[c];
    unsigned long long run = block_exclusive_scan(s, sh);
    for (long long c = hi - 1; c >= lo; --c) {
        alive[c] = run;
        run += hist[c];
    }
    __syncthreads();
    // base[k] = sum_{k' < k} alive[k'], segments in forward order
    const long long flo = (long long)threadIdx.x * seg, fhi = flo + seg < len ? flo + seg : len;
    s = 0;
    for (long long c = flo; c < fhi; ++c) s += alive[c];
    run = block_exclusive_scan(s, sh);
    for (long long c = flo; c < fhi; ++c) {
        base[c] = run;
        run += alive[c];
    }
    if (fhi == len && flo < fhi) {
        if (marg) {   // one warp per item; whole edges in the order of edge_item_key, else passes of chunks
            ctr->total_items[cls] = ctr->whole ? ctr->n_edges[cls] : base[maxc];
            ctr->next_item[cls] = 0;
            return;
        }
        const unsigned long long W = base[maxc];
        ctr->total_items[cls] = W;
        ctr->next_item[cls] = 0;
        ctr->cost[cls] = choose_pool(sc, cls, W, ctr, mean_n, forced_group, split_stride, allow_split, need_marg);
    }
}

// Both classes at once: class c's order goes to sorted[class_base(c) ..], the
// same region its edges occupy, so the two never overlap.
__device__ __forceinline__ void place_edges(const ProblemDev* probs, const EdgeWork* edges, long long edge_cap,
                                            int nclass, const DepthCounters* ctr, const unsigned long long* alive0,
                                            unsigned long long* cursor0, const unsigned long long* alive1,
                                            unsigned long long* cursor1, int32_t* sorted, long long first,
                                            long long step)
{
    const int gs = ctr->gs;
    const bool whole = ctr->whole != 0;
    const long long E0 = (long long)ctr->n_edges[0];
    const long long E = E0 + (nclass > 1 ? (long long)ctr->n_edges[1] : 0);
    const long long b1 = class_base(ctr, 1, edge_cap);
    for (long long k = first; k < E; k += step) {
        const bool front = k < E0;
        const long long e = front ? k : k - E0;
        const long long cb = front ? 0 : b1;
        const EdgeWork w = edges[cb + e];
        const long long ch = whole ? edge_item_key(w.total, probs[w.prob].N, probs[w.prob].ar[w.i], probs[w.prob].ar[w.j]) : chunk_count(w.total, gs);
        const unsigned long long pos =
            front ? alive0[ch] + atomicAdd(&cursor0[ch], 1ULL) : alive1[ch] + atomicAdd(&cursor1[ch], 1ULL);
        sorted[cb + (long long)pos] = (int32_t)e;
    }
}

// --------------------------------------------------------------------------
// End-of-depth removal over the snapshot (bits: the adjacency bit matrix of
// fbn_turn.cuh too).
__device__ __forceinline__ void apply_edges(const ProblemDev* probs, const EdgeWork* edges,
                                            const unsigned long long* min_accept, long long edge_cap,
                                            const long long* binom, int32_t* sep_pool, long long sep_cap,
                                            DepthCounters* ctr, long long first, long long step,
                                            unsigned* bits = nullptr)
{
    const int d = ctr->d;
    const long long n0 = (long long)ctr->n_edges[0], n1 = (long long)ctr->n_edges[1];
    unsigned long long my_tests = 0, my_removed = 0, my_samples = 0;
    for (long long k = first; k < n0 + n1; k += step) {
        const long long e = k < n0 ? k : edge_cap - n1 + (k - n0);
        const EdgeWork w = edges[e];
        const unsigned long long ma = min_accept[e];
        const bool rm = ma < (unsigned long long)w.total;
        const unsigned long long t = rm ? ma + 1 : (unsigned long long)w.total;
        my_tests += t;
        my_samples += t * (unsigned long long)probs[w.prob].N;
        if (!rm) continue;
        my_removed += 1;
        const ProblemDev P = probs[w.prob];
        const long long n = P.n;
        P.adj[w.i * n + w.j] = 0;
        P.adj[w.j * n + w.i] = 0;
        if (bits) {
            atomicAnd(bits + w.i * 4 + (w.j >> 5), ~(1u << (w.j & 31)));
            atomicAnd(bits + w.j * 4 + (w.i >> 5), ~(1u << (w.i & 31)));
        }
        long long off = 0;
        if (d > 0) {
            off = (long long)atomicAdd(&ctr->sep_used, (unsigned long long)d);
            if (off + d > sep_cap) {
                atomicOr(&ctr->status, kStatusSepPool);
                off = 0;
            } else {
                const bool xside = (long long)ma < w.cnt_i;
                const int a = xside ? w.i : w.j;
                const int posb = xside ? w.posj : w.posi;
                const long long lr = xside ? (long long)ma : (long long)ma - w.cnt_i;
                int pos[kMaxD];
                unrank_lex(lr, P.deg[a] - 1, d, binom, pos);
                const int32_t* nb = P.nbr + (long long)a * n;
                for (int q = 0; q < d; ++q) sep_pool[off + q] = nb[pos[q] < posb ? pos[q] : pos[q] + 1];
            }
        }
        P.sep_len[w.i * n + w.j] = d;
        P.sep_off[w.i * n + w.j] = off;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        my_tests += __shfl_xor_sync(0xffffffffu, my_tests, o);
        my_removed += __shfl_xor_sync(0xffffffffu, my_removed, o);
        my_samples += __shfl_xor_sync(0xffffffffu, my_samples, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (my_tests) atomicAdd(&ctr->tests_oracle, my_tests);
        if (my_samples) atomicAdd(&ctr->test_samples, my_samples);
        if (my_removed) atomicAdd(&ctr->removed, my_removed);
    }
}

// End of a depth (one CTA): record it; stop when it had no edge to test (no
// edge has a side with at least d candidates), when an error bit is set, or
// when the next depth exceeds max_depth (>= 0); clear the per-depth counters,
// the chunk histograms and the placement cursors for the next depth
// (clear_ends: the degree sum too).
__device__ __forceinline__ void depth_end(DepthCounters* ctr, DepthRecord* rec, int max_depth,
                                          unsigned long long* hist, unsigned long long* cursor, bool clear_ends)
{
    __shared__ long long used[2];   // histogram / cursor entries this depth touched per class
    if (threadIdx.x < 2) used[threadIdx.x] = (long long)ctr->maxc[threadIdx.x] + 1;
    __syncthreads();
    if (threadIdx.x == 0) {
        const int d = ctr->d;
        const long long E = (long long)(ctr->n_edges[0] + ctr->n_edges[1]);
        if (d < kMaxDepthRecords) {
            rec[d].edges = E;
            rec[d].tests = (long long)ctr->tests;
            rec[d].tests_oracle = (long long)ctr->tests_oracle;
            rec[d].test_samples = (long long)ctr->test_samples;
            rec[d].popc_work = (long long)ctr->popc_work;
            rec[d].smem_updates = (long long)ctr->smem_updates;
            rec[d].removed = (long long)ctr->removed;
            rec[d].t_end = gtime();
        }
        const int next = d + 1;
        const bool stop = E == 0 || ctr->status != 0 || (max_depth >= 0 && next > max_depth) || next > kMaxD ||
                          next >= kMaxDepthRecords;
        for (int c = 0; c < 2; ++c)
            ctr->n_edges[c] = ctr->maxc[c] = ctr->next_item[c] = ctr->total_items[c] = ctr->max_cells[c] = 0;
        ctr->tests = ctr->tests_oracle = ctr->removed = ctr->test_samples = ctr->popc_work = ctr->smem_updates = 0;
        ctr->gsel = 0;
        if (clear_ends) ctr->adj_ends = 0;
        ctr->nbr_claim = 0;
        ctr->max_total[0] = ctr->max_total[1] = 0;
        ctr->split[0] = ctr->split[1] = 1;
        ctr->cost[0] = ctr->cost[1] = 0.0f;
        ctr->whole = 0;
        ctr->direct = 0;
        ctr->d = next;
        __threadfence();
        ctr->active = stop ? 0 : 1;
    }
    for (int c = 0; c < 2; ++c) {
        const long long n = used[c] < kMaxPasses + 1 ? used[c] : kMaxPasses + 1;
        unsigned long long* hc = hist + c * (kMaxPasses + 1);
        unsigned long long* cc = cursor + c * (kMaxPasses + 1);
        for (long long k = threadIdx.x; k < n; k += blockDim.x) {
            hc[k] = 0;
            cc[k] = 0;
        }
    }
}

}  // namespace fbn
