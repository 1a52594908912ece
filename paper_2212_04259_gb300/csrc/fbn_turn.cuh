// fbn_turn.cuh -- from one depth to the next of a small problem, by one CTA.
//
// The persistent loop's way between two depths -- removal, snapshot, edge list,
// ordering, each behind a barrier of the whole grid -- took 22 of the 37 us of a
// small problem's depth.  For one problem of at most kTurnVertices variables
// the CTA that arrives last at the end of the tests does all of it: the
// adjacency is a bit matrix in shared memory (a neighbour's position is a
// popcount) and the edges of the next depth are listed from it.  Their order
// needs no histogram: item w is chunk w / E of edge w mod E, so that every edge
// gets its k-th chunk before any gets its (k+1)-th, and the items past an edge's
// last chunk are empty.  A depth of too many items is left to the general phases.
#pragma once

#include "fbn_graph.cuh"
#include "fbn_loop.h"

namespace fbn {

constexpr int kTurnWords = kTurnVertices / 32;
constexpr int kTurnPairs = kTurnVertices * (kTurnVertices - 1) / 2;

struct TurnShared {
    unsigned old_bits[kTurnVertices][kTurnWords];   // the snapshot the tests ran on
    unsigned bits[kTurnVertices][kTurnWords];
    int deg[kTurnVertices];
    long long sets[kTurnVertices];                  // C(k, next depth)
    int ar[kTurnVertices];
    unsigned short pair[kTurnPairs];                // the live edges: i << 8 | j
    unsigned long long tests, sep_base;
    unsigned max_cells[2], max_total[2];
    int removed, live, edges[2], at[2], items[2], chunks[2], too_big, heavy;
};

// The slot-th set bit of a row.
__device__ __forceinline__ int nth_neighbour(const unsigned* row, int slot)
{
    for (int w = 0; w < kTurnWords; ++w) {
        unsigned m = row[w];
        const int c = __popc(m);
        if (slot < c) {
            while (slot-- > 0) m &= m - 1;
            return w * 32 + __ffs(m) - 1;
        }
        slot -= c;
    }
    return 0;   // not reached: slot < degree
}

__device__ __forceinline__ int row_degree(const unsigned* row)
{
    int c = 0;
#pragma unroll
    for (int w = 0; w < kTurnWords; ++w) c += __popc(row[w]);
    return c;
}

// Place of neighbour j in its ascending row.
__device__ __forceinline__ int row_slot(const unsigned* row, int j)
{
    int c = __popc(row[j >> 5] & ((1u << (j & 31)) - 1u));
    for (int w = 0; w < (j >> 5); ++w) c += __popc(row[w]);
    return c;
}

// The kernels of a depth take over at depth ctr->d (one CTA, the others waiting): a
// table did not fit, or the depth is long enough for their speed to show.  Nothing of
// the depth is removed, and its state is as before its edge list.  Tests made stay
// counted.
__device__ __noinline__ void hand_over(const LoopArgs& a, DepthCounters* ctr)
{
    const long long used[2] = {(long long)ctr->maxc[0] + 1, (long long)ctr->maxc[1] + 1};
    __syncthreads();
    for (int c = 0; c < 2; ++c)
        for (long long k = threadIdx.x; k < used[c]; k += kTestThreads) a.hist[c * a.ord_cap + k] = a.cursor[c * a.ord_cap + k] = 0;
    if (threadIdx.x == 0) {
        for (int c = 0; c < 2; ++c)
            ctr->n_edges[c] = ctr->maxc[c] = ctr->next_item[c] = ctr->total_items[c] = ctr->max_cells[c] = ctr->max_total[c] = 0;
        const bool split = ctr->split[0] > 1 || ctr->split[1] > 1;
        ctr->split[0] = ctr->split[1] = 1;
        ctr->active = -1;
        ctr->adj_ends = 0;
        ctr->gsel = ctr->whole = ctr->direct = 0;
        *((volatile unsigned*)a.left) = kLoopHandedOver + (unsigned)ctr->d + (split ? kLoopSplit : 0u);
    }
}

// From this estimate of a depth's tests on the pools' own kernels win back a hand-over,
// which costs some 80 us: their rows have more L1, and up to kLoopOneCta variables
// twice the CTAs.  In the loop and handed over: 60 binary variables x 3,000 samples to
// depth 3 375 and 318 ms, 30 of them 24.1 and 11.0, depth 1 of 25 variables of 16 values
// x 100,000 (estimate 6.0e5), X^2, 1.67 and 1.28; depth 0 of 512 variables, 5.4e5, stays.
// choose_pool counts every rank; the edges that the depth before left say how many are
// tested (511 variables x 150 samples, 94% removed at depth 0: 20,235 of 579,390).
constexpr float kLoopHeavy = 5.7e5f;   // cycles

__device__ __forceinline__ bool depth_is_heavy(float cost, int d, const DepthRecord* rec)
{
    if (!(cost > kLoopHeavy) || d == 0 || d >= kMaxDepthRecords) return cost > kLoopHeavy;
    const float edges = (float)rec[d - 1].edges;
    return cost * (edges - (float)rec[d - 1].removed) > kLoopHeavy * edges;
}

// After the tests of depth ctr->d (apply: its removals are still to be made,
// the depth's items having been listed here), the whole CTA.
__device__ __noinline__ void turn(const LoopArgs& a, TurnShared& T, bool apply, int warps)
{
    DepthCounters* ctr = a.ctr;
    const ProblemDev& P = a.probs[0];
    const int n = P.n, tid = threadIdx.x, d = ctr->d;
    const long long n0 = (long long)ctr->n_edges[0], n1 = (long long)ctr->n_edges[1];
    const unsigned long long begin = gtime();
    for (int k = tid; k < kTurnVertices * kTurnWords; k += kTestThreads) {
        const unsigned w = a.bits[k];
        (&T.old_bits[0][0])[k] = w;
        (&T.bits[0][0])[k] = w;
    }
    if (tid < n) {
        T.ar[tid] = P.ar[tid];
        T.sets[tid] = binom_sat(a.binom, a.brows, tid, d + 1);
    }
    if (tid < 2) {
        T.edges[tid] = T.at[tid] = T.items[tid] = T.chunks[tid] = 0;
        T.max_cells[tid] = T.max_total[tid] = 0;
    }
    if (tid == 0) {
        T.tests = 0;
        T.removed = T.live = T.too_big = T.heavy = 0;
        T.sep_base = ctr->sep_used;
    }
    __syncthreads();
    if (apply) {
        unsigned long long tests = 0;
        for (long long k = tid; k < n0 + n1; k += kTestThreads) {
            const long long e = k < n0 ? k : a.edge_cap - n1 + (k - n0);
            const EdgeWork w = a.edges[e];
            const unsigned long long ma = a.min_accept[e];
            const bool rm = ma < (unsigned long long)w.total;
            tests += rm ? ma + 1 : (unsigned long long)w.total;
            if (!rm) continue;
            const int nth = atomicAdd(&T.removed, 1);
            atomicAnd(&T.bits[w.i][w.j >> 5], ~(1u << (w.j & 31)));
            atomicAnd(&T.bits[w.j][w.i >> 5], ~(1u << (w.i & 31)));
            P.adj[w.i * n + w.j] = 0;
            P.adj[w.j * n + w.i] = 0;
            long long off = 0;
            if (d > 0) {
                off = (long long)T.sep_base + (long long)nth * d;
                if (off + d > a.sep_cap) {
                    atomicOr(&ctr->status, kStatusSepPool);
                    off = 0;
                } else {
                    const bool xside = (long long)ma < w.cnt_i;
                    const int v = xside ? w.i : w.j, posb = xside ? w.posj : w.posi;
                    int pos[kMaxD];
                    unrank_lex(xside ? (long long)ma : (long long)ma - w.cnt_i, row_degree(T.old_bits[v]) - 1, d, a.binom, pos);
                    for (int q = 0; q < d; ++q)
                        a.sep_pool[off + q] = nth_neighbour(T.old_bits[v], pos[q] < posb ? pos[q] : pos[q] + 1);
                }
            }
            P.sep_len[w.i * n + w.j] = d;
            P.sep_off[w.i * n + w.j] = off;
        }
        if (tests) atomicAdd(&T.tests, tests);
        __syncthreads();
        if (tid == 0) {
            ctr->tests_oracle = T.tests;
            ctr->test_samples = T.tests * (unsigned long long)P.N;
            ctr->removed = T.removed;
            ctr->sep_used = T.sep_base + (unsigned long long)T.removed * d;
        }
    }
    __syncthreads();
    depth_end(ctr, a.rec, a.max_depth, a.hist, a.cursor, true);
    __syncthreads();
    const bool go = ctr->active != 0;
    // the snapshot of the next depth
    for (int k = tid; k < kTurnVertices * kTurnWords; k += kTestThreads) a.bits[k] = (&T.bits[0][0])[k];
    if (tid < n) {
        const int c = row_degree(T.bits[tid]);
        T.deg[tid] = c;
        P.deg[tid] = c;
    }
    for (int k = tid; k < n * kTurnWords; k += kTestThreads) {   // one word of a row
        const int v = k / kTurnWords, w = k - v * kTurnWords;
        int slot = 0;
        for (int q = 0; q < w; ++q) slot += __popc(T.bits[v][q]);
        for (unsigned m = T.bits[v][w]; m; m &= m - 1) P.nbr[(long long)v * n + slot++] = w * 32 + __ffs(m) - 1;
    }
    __syncthreads();
    if (!go) return;
    const int nd = d + 1;
    const bool marg = nd == 1 && a.marg1;
    // the live edges i < j, one place each
    for (int k = tid; k < n * kTurnWords; k += kTestThreads) {
        const int i = k / kTurnWords, w = k - i * kTurnWords;
        if (w < (i >> 5)) continue;
        unsigned m = T.bits[i][w];
        if (w == (i >> 5)) m &= ~((2u << (i & 31)) - 1u);   // j > i
        if (!m) continue;
        int at = atomicAdd(&T.live, __popc(m));
        for (; m; m &= m - 1) T.pair[at++] = (unsigned short)(i << 8 | (w * 32 + __ffs(m) - 1));
    }
    __syncthreads();
    const int live = T.live;
    const int gs = a.gs_forced > 0 ? a.gs_forced
                   : marg          ? (live >= warps ? kMargChunk : 1)
                                   : (live >= a.gs_edges ? 4 : 1);
    auto cells_of = [&](int i, int j) {
        unsigned long long cells = (unsigned long long)T.ar[i] * T.ar[j];
        for (int q = 0; q < nd && cells <= (unsigned long long)kMaxCells; ++q) cells *= (unsigned long long)P.max_arity;
        return cells < (1ull << 31) ? (unsigned)cells : 1u << 31;   // above kMaxCells: too big either way
    };
    // edges with a test: how many, their largest table and rank count, by class
    for (int k0 = 0; k0 < live; k0 += kTestThreads) {
        const int k = k0 + tid;
        int c = -1, chunks = 0;
        unsigned cells = 0, total = 0;
        if (k < live) {
            const int i = T.pair[k] >> 8, j = T.pair[k] & 255;
            const long long t = T.sets[T.deg[i] - 1] + T.sets[T.deg[j] - 1];
            if (t > kTurnItems * (long long)gs) {
                T.too_big = 1;
            } else if (t > 0) {
                cells = cells_of(i, j);
                c = (long long)cells <= a.warp_cells_cap ? 0 : 1;
                total = (unsigned)t;
                chunks = (int)chunk_count(t, gs);
            }
        }
        for (int q = 0; q < 2; ++q) {
            const unsigned in = __ballot_sync(0xffffffffu, c == q);
            if (!in) continue;
            const unsigned mc = __reduce_max_sync(0xffffffffu, c == q ? cells : 0u);
            const unsigned mt = __reduce_max_sync(0xffffffffu, c == q ? total : 0u);
            const int mk = (int)__reduce_max_sync(0xffffffffu, c == q ? (unsigned)chunks : 0u);
            const int sum = (int)__reduce_add_sync(0xffffffffu, c == q ? (unsigned)chunks : 0u);
            if ((tid & 31) == 0) {
                atomicAdd(&T.edges[q], __popc(in));
                atomicAdd(&T.items[q], sum);
                atomicMax(&T.max_cells[q], mc);
                atomicMax(&T.max_total[q], mt);
                atomicMax(&T.chunks[q], mk);
            }
        }
    }
    __syncthreads();
    const int E0 = T.edges[0], E1 = T.edges[1];
    const long long W[2] = {(long long)E0 * T.chunks[0], (long long)E1 * T.chunks[1]};
    if (T.too_big || W[0] > kTurnItems || W[1] > kTurnItems) return;   // general phases
    if (E0 + E1 == 0) {
        if (tid == 0) ctr->active = 0;   // no edge has a side with enough candidates
        return;
    }
    for (int k = tid; k < live; k += kTestThreads) {
        const int i = T.pair[k] >> 8, j = T.pair[k] & 255;
        const long long ci = T.sets[T.deg[i] - 1], total = ci + T.sets[T.deg[j] - 1];
        if (total <= 0) continue;
        const int c = (long long)cells_of(i, j) <= a.warp_cells_cap ? 0 : 1;
        const int at = atomicAdd(&T.at[c], 1);
        const long long e = c == 0 ? at : a.edge_cap - 1 - at;
        EdgeWork w;
        w.prob = 0;
        w.i = i;
        w.j = j;
        w.posj = (int16_t)row_slot(T.bits[i], j);
        w.posi = (int16_t)row_slot(T.bits[j], i);
        w.cnt_i = ci;
        w.total = total;
        a.edges[e] = w;
        a.min_accept[e] = (unsigned long long)total;
    }
    if (tid == 0) {
        float cost = 0.0f;
        ctr->n_edges[0] = E0;
        ctr->n_edges[1] = E1;
        ctr->gs = gs;
        ctr->whole = 0;
        ctr->direct = 1;
        for (int c = 0; c < 2; ++c) {
            ctr->max_cells[c] = T.max_cells[c];
            ctr->max_total[c] = T.max_total[c];
            ctr->next_item[c] = 0;
            ctr->total_items[c] = (unsigned long long)W[c];
            if (W[c] > 0 && !marg) {   // by the items that hold a test
                cost += choose_pool(a.sc[c], c, (unsigned long long)T.items[c], ctr, a.mean_n, a.forced_group, a.split_stride,
                            W[c] <= kSplitItems, a.need_marg);
                ctr->total_items[c] = (unsigned long long)W[c] * (unsigned long long)ctr->split[c];
            }
        }
        if (DepthRecord* r = nd < kMaxDepthRecords ? a.rec + nd : nullptr) {
            r->t_begin = begin;
            r->t_tests = gtime();
        }
        T.heavy = depth_is_heavy(cost, nd, a.rec);
    }
    __syncthreads();
    if (T.heavy) hand_over(a, ctr);
}

}  // namespace fbn
