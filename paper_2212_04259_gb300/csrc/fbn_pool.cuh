// fbn_pool.cuh -- device code of the per-depth CI-level work pool (Section
// IV-B) and of the edge-level form (Section IV-A): per-group state, the set-up
// of one conditioning set (Section IV-C), counting, the bounded decision,
// sample-split tests and the pool loop.  Each pool kernel is defined in its
// own translation unit (fbn_pool_small.cu, _big.cu, _mid.cu, fbn_plain.cu;
// depth 1 from one-hot planes in fbn_pool_marg.cu), so that they compile in
// parallel.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "fbn_depth.cuh"

namespace fbn {

// --------------------------------------------------------------------------
// Per-group state of a worker, in shared memory.
struct GroupState {
    long long r0, r1;
    unsigned long long tests;
    unsigned long long smem_updates;   // counting work done, flushed with tests
    unsigned long long item;   // split tests: the test's item and this group's part
    int part;
    unsigned ticket;
    int e;
    int go;
    double crit;       // exact critical value, 0 until the exact decision needs it
    float crit_lo, crit_hi;
    long long crit_q;  // floor(crit / 2) of the n ln n decision
    int pos[kMaxD];
};

// Fill the test of rank rk of edge w into the group's TestSpec.  Rank 0 of
// the group computes the subset positions (unranked when `fresh`, else the
// successor of the previous rank of the same side); one thread per
// conditioning variable then resolves its row.  Returns false (uniformly)
// when the table is over the cell limit.
template <int G>
__device__ __forceinline__ bool setup_rank(const ProblemDev& P, const EdgeWork& w, int d, long long rk, bool fresh,
                                           GroupState& S, const long long* binom, TestSpec& spec, unsigned* status)
{
    const int r = Grp<G>::rank();
    const bool xside = rk < w.cnt_i;
    const int a = xside ? w.i : w.j;
    const int posb = xside ? w.posj : w.posi;
    if (r == 0) {
        if (d > 0) {
            const long long lr = xside ? rk : rk - w.cnt_i;
            const int p = P.deg[a] - 1;
            if (fresh || lr == 0) unrank_lex(lr, p, d, binom, S.pos);
            else next_subset(p, d, S.pos);
        }
        spec.nrows = d + 2;
        spec.N = P.N;
    }
    Grp<G>::sync();
    if (r < d + 2) {
        int v;
        if (r < d) {
            const int t = S.pos[r];
            v = P.nbr[(long long)a * P.n + (t < posb ? t : t + 1)];
        } else {
            v = r == d ? w.i : w.j;
            if (r == d) spec.rx = P.ar[v]; else spec.ry = P.ar[v];
        }
        spec.rows[r] = P.data + (long long)v * P.ld;
        spec.rad[r] = P.ar[v];
    }
    Grp<G>::sync();
    long long cells = 1;
    for (int k = 0; k < d + 2 && cells <= kMaxCells; ++k) cells *= spec.rad[k];
    if (cells > kMaxCells) {
        if (r == 0) atomicOr(status, kStatusTooBig);
        return false;
    }
    if (r == 0) spec.cells = cells;
    Grp<G>::sync();
    return true;
}

// The decision of a counted test from its table and marginals: df from the
// declared arities or from the observed table (no degree of freedom left:
// the test cannot reject), crit from the cache, then the bounded statistic.
// In line: as a call it kept a fifth of the small tests' time (depth 2 of 40
// variables of 5 values x 1,000 samples, X^2: 7.2 -> 5.8 ms).
template <int G>
__device__ __forceinline__ int decide_test(const PoolArgs& a, const TestSpec& spec, const int* T, int* M,
                                        GroupState& S, double* red, unsigned* status)
{
    grp_marginals<G>(spec, T, M);
    const int nz = (int)spec.cells / (spec.rx * spec.ry);   // cells <= kMaxCells < 2^31: 32-bit
    const long long df = a.df_mode ? grp_df_adjusted<G>(spec, M, red)
                                   : (long long)((spec.rx - 1) * (spec.ry - 1)) * nz;
    if (Grp<G>::rank() == 0) {
        // the float bracket of crit when the table has it; else the exact
        // value (computed and stored on first use) and its bracket
        float2 f = make_float2(0.0f, 0.0f);
        if (df > 0 && df < a.crit.dense_n) f = a.crit.dense_f[df];
        S.crit = 0.0;
        if (df > 0 && !(f.y > 0.0f)) {
            const double c = crit_get(a.crit, df, a.alpha, status);
            S.crit = c;
            f = make_float2(__double2float_rd(c), __double2float_ru(c));
        }
        S.crit_lo = f.x;
        S.crit_hi = f.y;
        S.tests += 1;   // flushed to the depth counter when the group leaves the pool
    }
    Grp<G>::sync();
    if (df <= 0) return 1;   // p = 1 > alpha
    const int dec = grp_decide_bound<G>(spec, T, M, S.crit_lo, S.crit_hi, red, a.stat);
    if (dec >= 0) return dec;
    // the band straddles crit: exact FP64 statistic against the exact value
    if (Grp<G>::rank() == 0 && S.crit == 0.0) S.crit = crit_get(a.crit, df, a.alpha, status);
    Grp<G>::sync();
    const double ex = a.stat == kStatX2 ? grp_x2_exact<G>(spec, T, M, red) : grp_g2_exact<G>(spec, T, M, red);
    return ex < S.crit ? 1 : 0;
}

// G^2 with the declared df from the n ln n table; FP64 when the error bound
// straddles crit.
template <int G>
__device__ __forceinline__ int decide_lut(const PoolArgs& a, const TestSpec& spec, const int* T, GroupState& S,
                                          double* red, unsigned* status)
{
    const int nz = (int)spec.cells / (spec.rx * spec.ry);
    const long long df = (long long)((spec.rx - 1) * (spec.ry - 1)) * nz;
    if (Grp<G>::rank() == 0) {
        long long q = df < a.crit.dense_n ? a.crit.dense_q[df] : 0;
        if (q == 0) q = (long long)floor(crit_get(a.crit, df, a.alpha, status) * 0.5 * 68719476736.0);   // 2^kLutBits
        S.crit_q = q;
        S.tests += 1;   // flushed to the depth counter when the group leaves the pool
    }
    const long long g = grp_g2_lut<G>(spec, T, a.lut, red);
    Grp<G>::sync();
    const long long q = S.crit_q;
    const long long err = a.lut_err * ((long long)spec.cells + (long long)nz * (spec.rx + spec.ry + 1));
    if (g + err < q) return 1;
    if (g - err > q) return 0;   // q + 1 bounds crit from above
    const double ex = grp_g2_cells<G>(spec, T, red);
    if (Grp<G>::rank() == 0) S.crit = crit_get(a.crit, df, a.alpha, status);
    Grp<G>::sync();
    return ex < S.crit ? 1 : 0;
}

// Counting work of one table (rank 0): one shared-memory update per sample.
template <int G>
__device__ __forceinline__ void note_work(GroupState& S, const TestSpec& spec)
{
    if (Grp<G>::rank() != 0) return;
    S.smem_updates += (unsigned long long)spec.N;
}

// Run one rank: 1 = accepts independence, 0 = rejects, -1 = could not run.
template <int G>
__device__ __forceinline__ int run_rank(const PoolArgs& a, int d, const ProblemDev& P, const EdgeWork& w, long long rk,
                                        bool fresh, GroupState& S, TestSpec& spec, int* slice, long long slice_ints,
                                        int* gtab, double* red)
{
    unsigned* status = &a.ctr->status;
    if (!setup_rank<G>(P, w, d, rk, fresh, S, a.binom, spec, status)) return -1;
    int* M = nullptr;
    const int* T = grp_table<G>(spec, slice, slice_ints, gtab, a.gscratch_ints, a.lut == nullptr, &M);
    if (!T) {
        if (Grp<G>::rank() == 0) {
            if (a.hand_over) {   // the kernels of a depth take it from here: no further claims
                *((volatile int*)&a.ctr->hand_over) = 1;
                for (int c = 0; c < 2; ++c) atomicAdd(&a.ctr->next_item[c], 1ULL << 40);
            } else {   // the global scratch is too small: the host grows it and starts over
                atomicOr(status, kStatusScratch);
                atomicMax(&a.ctr->need_cells, (int)spec.cells);
            }
        }
        return -1;
    }
    note_work<G>(S, spec);
    return a.lut ? decide_lut<G>(a, spec, T, S, red, status) : decide_test<G>(a, spec, T, M, S, red, status);
}

// One part of a split test: count samples [N p / S, N (p + 1) / S) (16-aligned
// bounds) of rank rk into the test's global table; the part that finishes last
// copies the table into shared memory (L2 reads), zeroes it, decides and
// lowers the edge's rank.  Returns 1 when this group decided an acceptance.
template <int G>
__device__ __noinline__ int run_split_part(const PoolArgs& a, int d, const ProblemDev& P, const EdgeWork& w,
                                              long long rk, int split, GroupState& S, TestSpec& spec, int* slice,
                                              long long slice_ints, int* gtab, double* red,
                                              const unsigned long long* min_accept_e)
{
    unsigned* status = &a.ctr->status;
    const int r = Grp<G>::rank();
    int* Tg = a.split_tab + (long long)S.item * a.split_stride;
    if (r == 0) S.go = (unsigned long long)rk <= *((volatile const unsigned long long*)min_accept_e);
    Grp<G>::sync();
    bool ready = false;   // spec holds this rank's table shape (uniform over the group)
    if (S.go && setup_rank<G>(P, w, d, rk, true, S, a.binom, spec, status)) {
        ready = true;
        const long long N = P.N;
        // part bounds on 128-sample boundaries: whole 16-byte vectors
        const long long lo = (N * S.part / split) & ~127LL;
        const long long hi = S.part == split - 1 ? N : ((N * (S.part + 1) / split) & ~127LL);
        if (r < d + 2) spec.rows[r] += lo;
        Grp<G>::sync();
        if (r == 0) spec.N = (int)(hi - lo);
        Grp<G>::sync();
        int* M = nullptr;
        const int* T = grp_table<G>(spec, slice, slice_ints, gtab, a.gscratch_ints, a.lut == nullptr, &M);
        if (!T) {
            if (r == 0) {
                atomicOr(status, kStatusScratch);
                atomicMax(&a.ctr->need_cells, (int)spec.cells);
            }
        } else {
            note_work<G>(S, spec);
            for (long long c = r; c < spec.cells; c += G)
                if (T[c]) atomicAdd(Tg + c, T[c]);
        }
    }
    __threadfence();
    Grp<G>::sync();
    if (r == 0) S.ticket = atomicAdd(&a.split_ticket[S.item], 1u);
    Grp<G>::sync();
    if (S.ticket != (unsigned)(split - 1)) return 0;
    // the last part: every other part's adds are in L2; the decision needs
    // the table's shape only (cells, radices), which this part's own setup
    // left in spec when it counted
    __threadfence();
    if (!ready && !setup_rank<G>(P, w, d, rk, true, S, a.binom, spec, status)) return 0;
    const long long C = spec.cells;
    int* Tl = slice;
    for (long long c = r; c < C; c += G) {
        Tl[c] = __ldcg(Tg + c);
        Tg[c] = 0;
    }
    if (r == 0) {
        spec.N = P.N;   // the table holds every part's samples
        a.split_ticket[S.item] = 0;
        S.go = (unsigned long long)rk <= *((volatile const unsigned long long*)min_accept_e);
    }
    Grp<G>::sync();
    if (!S.go) return 0;
    return a.lut ? decide_lut<G>(a, spec, Tl, S, red, status)
                 : decide_test<G>(a, spec, Tl, Tl + C, S, red, status);
}

// Shared state of a pool CTA, sized for the most groups per CTA (8 warps), and
// what a claim needs of the depth (kept here, not in every thread's registers:
// the counting loops use all of them).
struct PoolShared {
    TestSpec spec[kTestThreads / 32];
    GroupState st[kTestThreads / 32];
    double red[32];
    unsigned long long total, groups;   // items of the class; items taken without a claim
    long long cb, maxc;                 // the class's first edge, its passes
    const unsigned long long* base;     // first item of each pass
    unsigned edges;                     // edges of the class when the items are laid out directly, else 0
    int gs, split;
    unsigned long long pass_base[kBaseSmem];
};

// One thread of a group: item wi, or for ~0 the next one of the counter, into S
// (e = -1: none left).
static __device__ __noinline__ void claim_item(const PoolArgs& a, const PoolShared& sh, GroupState& S,
                                               unsigned long long wi)
{
    if (wi == ~0ULL)
        wi = sh.total > sh.groups ? sh.groups + atomicAdd(&a.ctr->next_item[a.cls], 1ULL) : sh.total;
    S.e = -1;
    if (wi >= sh.total) return;
    const unsigned long long w = sh.split == 1 ? wi : wi / (unsigned long long)sh.split;
    S.item = w;
    S.part = (int)(wi - w * (unsigned long long)sh.split);
    long long pass;
    int e;
    if (sh.edges) {   // w < 2^31
        pass = (unsigned)w / sh.edges;
        e = (int)((unsigned)w - (unsigned)pass * sh.edges);
    } else {
        long long lo = 0, hi = sh.maxc - 1;   // largest pass with base[pass] <= w
        while (lo < hi) {
            const long long mid = (lo + hi + 1) >> 1;
            if (sh.base[mid] <= w) lo = mid; else hi = mid - 1;
        }
        pass = lo;
        e = a.sorted[sh.cb + (long long)(w - sh.base[lo])];
    }
    const long long tot = a.edges[sh.cb + e].total;
    const long long cr = chunk_ranks(tot, sh.gs);
    const long long r0 = pass * cr;
    S.e = e;
    S.r0 = r0;
    S.r1 = r0 + cr < tot ? r0 + cr : tot;
}

// LOOP: in the persistent loop a group's first item is its own index and the
// later ones come from the counter (no claim at all with fewer items than
// groups: one round trip less on a small problem's critical path).
template <int G, bool LOOP = false>
__device__ __forceinline__ void pool_body(const PoolArgs& a, int* smem, PoolShared& sh)
{
    constexpr int NG = G >= kTestThreads ? 1 : kTestThreads / G;   // groups per CTA
    const int d = a.ctr->d;
    if (a.ctr->total_items[a.cls] == 0) return;
    const int g = Grp<G>::gid();
    const int r = Grp<G>::rank();
    if (threadIdx.x == 0) {
        const DepthCounters* ctr = a.ctr;
        sh.total = ctr->total_items[a.cls];
        sh.groups = LOOP ? (unsigned long long)gridDim.x * NG : 0;
        sh.cb = class_base(ctr, a.cls, a.edge_cap);
        sh.maxc = (long long)ctr->maxc[a.cls];
        sh.edges = ctr->direct ? (unsigned)ctr->n_edges[a.cls] : 0u;
        sh.base = !sh.edges && sh.maxc + 1 <= kBaseSmem ? sh.pass_base : a.base;
        sh.gs = ctr->gs;
        sh.split = ctr->split[a.cls] > 1 ? ctr->split[a.cls] : 1;
    }
    __syncthreads();
    if (sh.base == sh.pass_base)
        for (long long k = threadIdx.x; k <= sh.maxc; k += blockDim.x) sh.pass_base[k] = a.base[k];
    const long long slice_ints = a.smem_ints / NG;
    int* slice = smem + g * slice_ints;
    int* gtab = a.gscratch ? a.gscratch + ((long long)blockIdx.x * NG + g) * a.gscratch_ints : nullptr;
    GroupState& S = sh.st[g];
    TestSpec& spec = sh.spec[g];
    if (r == 0) S.tests = S.smem_updates = 0;
    __syncthreads();

    for (bool first = LOOP;; first = false) {
        if (r == 0) claim_item(a, sh, S, first ? (unsigned long long)g * gridDim.x + blockIdx.x : ~0ULL);
        Grp<G>::sync();
        if (S.e < 0) break;
        const EdgeWork w = a.edges[sh.cb + S.e];
        const ProblemDev& P = a.probs[w.prob];
        unsigned long long* min_accept = a.min_accept + sh.cb + S.e;
        const long long r0 = S.r0, r1 = S.r1;
        if (r0 >= r1) {   // past the edge's last chunk
            Grp<G>::sync();
            continue;
        }
        if (sh.split > 1) {   // single-rank items (gs = 1, no edge above kMaxPasses ranks)
            const int res = run_split_part<G>(a, d, P, w, r0, sh.split, S, spec, slice, slice_ints, gtab, sh.red, min_accept);
            if (res == 1 && r == 0) atomicMin(min_accept, (unsigned long long)r0);
            Grp<G>::sync();
            continue;
        }
        for (long long rk = r0; rk < r1; ++rk) {
            if (r == 0) S.go = (unsigned long long)rk <= *((volatile unsigned long long*)min_accept);
            if (LOOP && r == 0 && rk > r0) atomicAdd(&a.ctr->beat, 1u);
            Grp<G>::sync();
            if (!S.go) break;
            const int res = run_rank<G>(a, d, P, w, rk, rk == r0, S, spec, slice, slice_ints, gtab, sh.red);
            if (res == 1 && r == 0) atomicMin(min_accept, (unsigned long long)rk);
            if (res != 0) break;
        }
        Grp<G>::sync();
    }
    if (r == 0 && S.tests) atomicAdd(&a.ctr->tests, S.tests);
    if (r == 0 && S.smem_updates) atomicAdd(&a.ctr->smem_updates, S.smem_updates);
}

// The end of a test CTA in the depth's record (the latest over CTAs).
__device__ __forceinline__ void tests_done(const DepthCounters* ctr)
{
    __syncthreads();
    if (threadIdx.x == 0)
        if (DepthRecord* r = depth_rec(ctr, ctr->d)) atomicMax(&r->t_tests_end, gtime());
}

}  // namespace fbn
