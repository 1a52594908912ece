// fbn_pool_marg.cuh -- the work pool of depth 1 for arities up to 5, and every
// pair's table at depth 0 for problems too small for the tensor-core Gram, by
// POPC over one-hot bit planes.
//
// Depth 0 leaves every pair's table in the Gram matrix, so of the table of
// (x, y | z) all three pair margins N_xy+, N_x+z, N_+yz are known before
// anything is counted.  Only the (r_x - 1)(r_y - 1)(r_z - 1) cells with x, y,
// z >= 1 are counted; every other cell follows from those and the margins by
// inclusion and exclusion.  For arities 2, 3, 4 in equal parts that is 8 counts
// per 32 samples on average where the whole table takes 27 (36 with loops of
// fixed length), and a byte histogram takes 32 shared-memory reductions.
//
// One-hot planes (built at upload, bit s of word w of plane a of variable v:
// sample 32 w + s has value a + 1; zero past the samples) make a cell and 32
// samples one LOP3 and one POPC.  A warp runs one test; the counters of a pass
// (one or two values of z) stay in registers, one REDUX per counter (or per two,
// packed, below 65,536 samples) adds them over the lanes, and lane 5 x + y ends
// with the cells (., x, y).  No shared memory, no marginal sums, no integer
// division: the margins of the statistic are the margins already loaded.
//
// The pool was bound by the latency and instructions of one test, not by its
// counting unit (5,200 instructions a test of 13,000 samples, of which 3,000
// outside the sample loop).  Measured, whole depth 1: see k_pool_marg.
#pragma once

#include "fbn_pool.cuh"

namespace fbn {
namespace {

constexpr int kMA = kMargMaxArity;

// sum over (a, b) of s_x(a) s_y(b) R(a, b) for lane (x, y): the inclusion and
// exclusion of the counted cells; s(a) = -1 at value 0, 1 at value a + 1, else 0
__device__ __forceinline__ int ie_sign(int value, int a)
{
    return value == 0 ? -1 : value == a + 1 ? 1 : 0;
}

// Counts of the cells (a, b, c) with A x-values, B y-values and C strata over
// the planes' 64-bit words, added over the warp and folded into this lane's
// cell of each stratum.
template <int A, int B, int C>
__device__ __forceinline__ int2 count_cells(const uint2* __restrict__ x, const uint2* __restrict__ y,
                                            const uint2* __restrict__ z, int ld2, int nw2, int lx, int ly, bool pack)
{
    const int lane = threadIdx.x & 31;
    unsigned acc[C][A][B];
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
        for (int a = 0; a < A; ++a)
#pragma unroll
            for (int b = 0; b < B; ++b) acc[c][a][b] = 0u;
    // the next word's planes are loaded while this one is counted
    uint2 X[A], Y[B], Z[C];
    int w = min(lane, nw2 - 1);
#pragma unroll
    for (int a = 0; a < A; ++a) X[a] = __ldg(x + a * ld2 + w);
#pragma unroll
    for (int b = 0; b < B; ++b) Y[b] = __ldg(y + b * ld2 + w);
#pragma unroll
    for (int c = 0; c < C; ++c) Z[c] = __ldg(z + c * ld2 + w);
#pragma unroll 1
    for (w = lane; w < nw2; w += 32) {
        uint2 U[A], V[B], W[C];
#pragma unroll
        for (int a = 0; a < A; ++a) U[a] = X[a];
#pragma unroll
        for (int b = 0; b < B; ++b) V[b] = Y[b];
#pragma unroll
        for (int c = 0; c < C; ++c) W[c] = Z[c];
        const int wn = min(w + 32, nw2 - 1);
#pragma unroll
        for (int a = 0; a < A; ++a) X[a] = __ldg(x + a * ld2 + wn);
#pragma unroll
        for (int b = 0; b < B; ++b) Y[b] = __ldg(y + b * ld2 + wn);
#pragma unroll
        for (int c = 0; c < C; ++c) Z[c] = __ldg(z + c * ld2 + wn);
#pragma unroll
        for (int c = 0; c < C; ++c)
#pragma unroll
            for (int a = 0; a < A; ++a)
#pragma unroll
                for (int b = 0; b < B; ++b)
                    acc[c][a][b] += __popc(U[a].x & V[b].x & W[c].x) + __popc(U[a].y & V[b].y & W[c].y);
    }
    int s[2] = {0, 0};
    if (pack && C == 2) {   // both strata's counts of a cell in one REDUX: each below 2^16
#pragma unroll
        for (int a = 0; a < A; ++a) {
            int u0 = 0, u1 = 0;
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const unsigned r = __reduce_add_sync(0xffffffffu, acc[0][a][b] | (acc[C - 1][a][b] << 16));
                const int sy = ie_sign(ly, b);
                u0 += sy * (int)(r & 0xFFFFu);
                u1 += sy * (int)(r >> 16);
            }
            const int sx = ie_sign(lx, a);
            s[0] += sx * u0;
            s[1] += sx * u1;
        }
    } else {
#pragma unroll
        for (int c = 0; c < C; ++c)
#pragma unroll
            for (int a = 0; a < A; ++a) {
                int u = 0;
#pragma unroll
                for (int b = 0; b < B; ++b)
                    u += ie_sign(ly, b) * (int)__reduce_add_sync(0xffffffffu, acc[c][a][b]);
                s[c] += ie_sign(lx, a) * u;
            }
    }
    return make_int2(s[0], s[1]);
}

// Strata per pass: two while the counters and words fit the register budget.
__device__ __forceinline__ int pass_strata(int A, int B, int left)
{
    return left >= 2 && A * B <= 6 ? 2 : 1;
}

// A >= B (the endpoint of larger arity is x): ten shapes, six of them with one
// or two strata.
__device__ __forceinline__ int2 count_shape(int A, int B, int C, const uint2* x, const uint2* y, const uint2* z,
                                            int ld2, int nw2, int lx, int ly, bool pack)
{
    switch ((A * 4 + B) * 2 + C) {
#define FBN_SHAPE(a, b, c) case ((a) * 4 + (b)) * 2 + (c): return count_cells<a, b, c>(x, y, z, ld2, nw2, lx, ly, pack)
        FBN_SHAPE(1, 1, 1); FBN_SHAPE(1, 1, 2);
        FBN_SHAPE(2, 1, 1); FBN_SHAPE(2, 1, 2);
        FBN_SHAPE(2, 2, 1); FBN_SHAPE(2, 2, 2);
        FBN_SHAPE(3, 1, 1); FBN_SHAPE(3, 1, 2);
        FBN_SHAPE(3, 2, 1); FBN_SHAPE(3, 2, 2);
        FBN_SHAPE(3, 3, 1);
        FBN_SHAPE(4, 1, 1); FBN_SHAPE(4, 1, 2);
        FBN_SHAPE(4, 2, 1);
        FBN_SHAPE(4, 3, 1);
        FBN_SHAPE(4, 4, 1);
#undef FBN_SHAPE
        default: return make_int2(0, 0);
    }
}

// What a warp knows of its edge and of one conditioning variable.
struct MargEdge {
    const uint2 *xp, *yp;   // planes of x and y
    const int32_t* gram;
    long long ld;           // row stride of the Gram
    int ox, oy;             // first Gram row of x and y
    int vx, vy;             // variables
    int rx, ry;
};

// Pair margin N(u = a, v = b) from the Gram's upper triangle.
__device__ __forceinline__ int pair_count(const int32_t* g, long long ld, int u, int ou, int a, int v, int ov, int b)
{
    return u < v ? g[(ou + a) * ld + ov + b] : g[(ov + b) * ld + ou + a];
}

// The decision in exact FP64 (the band straddled crit, or crit was not in the
// table) from the cells the test left in the warp's shared memory, T[z][lane].
// About one test in 1,000.  (Counting those tests again, cell by cell, made a
// single one of 100,000 samples last 2 ms.)
__device__ __noinline__ int marg_exact(const PoolArgs& a, const int* T, int rx, int ry, int rz)
{
    const int lane = threadIdx.x & 31, lx = lane / kMA, ly = lane - lx * kMA;
    const bool cell = lx < rx && ly < ry;
    double st = 0.0;
    long long df = 0;
    for (int z = 0; z < rz; ++z) {
        const int n = cell ? T[z * 32 + lane] : 0;
        int nx = 0, ny = 0;
        for (int q = 0; q < kMA; ++q) {
            nx += __shfl_sync(0xffffffffu, n, min(lx * kMA + q, 31));
            ny += __shfl_sync(0xffffffffu, n, min(q * kMA + ly, 31));
        }
        int nz = 0;
        for (int q = 0; q < kMA; ++q) nz += __shfl_sync(0xffffffffu, nx, q * kMA);
        if (cell) {
            const long long p = (long long)n * nz, q = (long long)nx * ny;
            if (a.stat == kStatX2) {
                if (q > 0) {
                    const double dd = (double)(p - q);
                    st += dd * dd / ((double)nz * (double)nx * (double)ny);
                }
            } else if (n > 0) {
                st += 2.0 * (double)n * log1p((double)(p - q) / (double)q);
            }
        }
        const int ax = __popc(__ballot_sync(0xffffffffu, cell && ly == 0 && nx > 0));
        const int ay = __popc(__ballot_sync(0xffffffffu, cell && lx == 0 && ny > 0));
        if (ax > 0 && ay > 0) df += (ax - 1) * (ay - 1);
    }
    if (!a.df_mode) df = (long long)(rx - 1) * (ry - 1) * rz;
    if (df <= 0) return 1;   // no degree of freedom left: p = 1
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) st += __shfl_xor_sync(0xffffffffu, st, o);
    int dec = 0;
    if (lane == 0) dec = st < crit_get(a.crit, df, a.alpha, &a.ctr->status);
    return __shfl_sync(0xffffffffu, dec, 0);
}

// One test (x, y | z): 1 accepts independence, 0 rejects.  nxy: N_xy+ of this
// lane's cell.
__device__ __forceinline__ int marg_test(const PoolArgs& a, const ProblemDev& P, const MargEdge& E, int vz, int rz,
                                         int oz, int nxy, int lx, int ly, int ld2, int nw2, int* T)
{
    const bool cx = lx < E.rx, cy = ly < E.ry, cell = cx && cy;
    const int N = P.N;
    const bool narrow = N < 65536;
    const uint2* zp = reinterpret_cast<const uint2*>(P.planes) + (long long)vz * P.nplanes * ld2;
    // margins of stratum z: N_x+z, N_+yz and N_++z
    const int32_t* gx = E.gram + (E.vx < vz ? (E.ox + lx) * E.ld + oz : (long long)oz * E.ld + E.ox + lx);
    const int32_t* gy = E.gram + (E.vy < vz ? (E.oy + ly) * E.ld + oz : (long long)oz * E.ld + E.oy + ly);
    const int32_t* gz = E.gram + oz * (E.ld + 1);
    const long long sx = E.vx < vz ? 1 : E.ld, sy = E.vy < vz ? 1 : E.ld, sz = E.ld + 1;
    // the float bracket of crit, read by lane 0 and broadcast: another warp
    // may be storing it, and every lane must take the same branch
    float2 cr = make_float2(0.0f, 0.0f);
    int df = (E.rx - 1) * (E.ry - 1) * rz;
    if (!a.df_mode && (threadIdx.x & 31) == 0) cr = a.crit.dense_f[df];
    int n0 = nxy, dfo = 0;
    float acc = 0.0f, mag = 0.0f;
    auto stratum = [&](int z, int n, int nx, int ny, int nz) {
        T[z * 32 + (threadIdx.x & 31)] = n;   // read back by this lane, in marg_exact
        if (cell && nx > 0 && ny > 0) marg_term(n, nz, nx, ny, narrow, a.stat, acc, mag);
        if (a.df_mode) {
            const int ax = __popc(__ballot_sync(0xffffffffu, cell && ly == 0 && nx > 0));
            const int ay = __popc(__ballot_sync(0xffffffffu, cell && lx == 0 && ny > 0));
            if (ax > 0 && ay > 0) dfo += (ax - 1) * (ay - 1);
        }
    };
    // the cell's part that the margins alone give
    auto known = [&](int nx, int ny, int nz) { return lx > 0 ? (ly > 0 ? 0 : nx) : (ly > 0 ? ny : nx + ny - nz); };
    const int mx0 = cx ? gx[0] : 0, my0 = cy ? gy[0] : 0, mz0 = gz[0];
    for (int c = 1; c < rz;) {
        const int C = pass_strata(E.rx - 1, E.ry - 1, rz - c);
        const int mx1 = cx ? gx[c * sx] : 0, my1 = cy ? gy[c * sy] : 0, mz1 = gz[c * sz];
        int mx2 = 0, my2 = 0, mz2 = 0;
        if (C == 2) {
            mx2 = cx ? gx[(c + 1) * sx] : 0;
            my2 = cy ? gy[(c + 1) * sy] : 0;
            mz2 = gz[(c + 1) * sz];
        }
        const int2 s = count_shape(E.rx - 1, E.ry - 1, C, E.xp, E.yp, zp + (long long)(c - 1) * ld2, ld2, nw2, lx, ly,
                                   narrow);
        const int t1 = cell ? known(mx1, my1, mz1) + s.x : 0;
        n0 -= t1;
        stratum(c, t1, mx1, my1, mz1);
        if (C == 2) {
            const int t2 = cell ? known(mx2, my2, mz2) + s.y : 0;
            n0 -= t2;
            stratum(c + 1, t2, mx2, my2, mz2);
        }
        c += C;
    }
    stratum(0, n0, mx0, my0, mz0);
    if (a.df_mode) {
        df = dfo;
        if (df <= 0) return 1;   // p = 1 > alpha
        if ((threadIdx.x & 31) == 0) cr = a.crit.dense_f[df];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_xor_sync(0xffffffffu, acc, o);
        mag += __shfl_xor_sync(0xffffffffu, mag, o);
    }
    int dec = -1;
    if (cr.y > 0.0f) dec = decide_from_sums(acc, mag, (float)kMA, 5.0f, a.stat, cr.x, cr.y, kMargTermRel);
    dec = __shfl_sync(0xffffffffu, dec, 0);   // lane 0 has the bracket
    return dec >= 0 ? dec : marg_exact(a, T, E.rx, E.ry, rz);
}

}  // namespace

// Depth 1 over the edges of every problem: one warp per item.  With many edges
// against the warps an item is a whole edge, the largest (tests x samples)
// first, its tests in order up to the first that accepts: as many tests as the
// sequential order runs.  With fewer an item is a chunk of consecutive ranks,
// pass by pass, as in the other pools.
//
// Measured on GB300, test window of depth 1 (before: two bit planes with every
// cell counted, or byte histograms): 256 problems of 20-300 variables 13.4 ->
// 5.4 ms, 20 of them 1.64 -> 0.62 ms, 1,000 variables x 100,000 samples (arities
// to 5) 3.92 -> 1.63 ms, 40 x 50,000 0.109 -> 0.036 ms.  1,130 instructions a test
// of 13,000 samples (5,200 before), issued in 46% of the cycles; the rest waits
// for the words and margins of the next pass.  What bounded it on the way:
// instruction fetch (16 inlined loops, edges in any order: 6 of 13 stall cycles
// without an instruction, 8.0 ms; the loops of one shape together: 6.0 ms), then
// the loads of a pass (the next word's planes in flight: 5.4 ms).  Two CTAs of
// 128 registers: three (80 registers, spills) 6.7 ms, five of 128 threads 6.2 ms.
// LOOP: in the persistent loop, where the items may be laid out directly and a
// warp's first item is its own index (a claim less on the critical path; with
// many items the counter's order is the better one: depth 1 of 20 problems 0.64
// against 0.68 ms).
template <bool LOOP>
__device__ __forceinline__ void marg_body(const PoolArgs& a)
{
    __shared__ unsigned long long s_base[kBaseSmem];
    __shared__ int s_cells[kMargThreads / 32][kMA * 32];   // a warp's table: [z][lane]
    const DepthCounters* ctr = a.ctr;
    const unsigned long long total = ctr->total_items[kClassWarp];
    if (total == 0) return;
    const int lane = threadIdx.x & 31, lx = lane / kMA, ly = lane - lx * kMA;
    const bool whole = ctr->whole != 0, direct = LOOP && ctr->direct != 0;
    const int gs = ctr->gs;
    const long long maxc = (long long)ctr->maxc[kClassWarp];
    const bool base_in_smem = !whole && !direct && maxc + 1 <= kBaseSmem;
    if (base_in_smem)
        for (long long k = threadIdx.x; k <= maxc; k += blockDim.x) s_base[k] = a.base[k];
    __syncthreads();
    const unsigned long long* base = base_in_smem ? s_base : a.base;
    unsigned long long tests = 0, work = 0;
    const unsigned long long all_warps = LOOP ? (unsigned long long)gridDim.x * (blockDim.x >> 5) : 0;
    bool first = LOOP;
    for (;;) {
        unsigned long long wi = (unsigned long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
        if (!first) {
            if (LOOP && total <= all_warps) break;
            if (lane == 0) wi = all_warps + atomicAdd(&a.ctr->next_item[kClassWarp], 1ULL);
            wi = __shfl_sync(0xffffffffu, wi, 0);
        }
        first = false;
        if (wi >= total) break;
        long long pass = 0;
        unsigned own = 0;
        if (direct) {
            const unsigned E = (unsigned)ctr->n_edges[kClassWarp];
            pass = (unsigned)wi / E;
            own = (unsigned)wi - (unsigned)pass * E;
        } else if (!whole) {   // largest pass with base[pass] <= wi
            long long lo = 0, hi = maxc - 1;
            while (lo < hi) {
                const long long mid = (lo + hi + 1) >> 1;
                if (base[mid] <= wi) lo = mid; else hi = mid - 1;
            }
            pass = lo;
        }
        const int e = direct ? (int)own : a.sorted[whole ? wi : wi - base[pass]];
        const EdgeWork w = a.edges[e];
        const ProblemDev& P = a.probs[w.prob];
        unsigned long long* min_accept = a.min_accept + e;
        const long long cr = whole ? w.total : chunk_ranks(w.total, gs);
        const int r0 = (int)(pass * cr), r1 = (int)(r0 + cr < w.total ? r0 + cr : w.total);
        if (!whole) {   // read by lane 0 and broadcast: other warps lower it, and the warp must stay together
            unsigned long long ma = 0;
            if (lane == 0) ma = *((volatile unsigned long long*)min_accept);
            if ((unsigned long long)r0 > __shfl_sync(0xffffffffu, ma, 0)) continue;
        }
        MargEdge E;
        const int ri = P.ar[w.i], rj = P.ar[w.j];
        E.vx = ri >= rj ? w.i : w.j;
        E.vy = ri >= rj ? w.j : w.i;
        E.rx = max(ri, rj);
        E.ry = min(ri, rj);
        E.ox = P.off[E.vx];
        E.oy = P.off[E.vy];
        E.gram = P.gram;
        E.ld = P.gram_ld;
        const int ld2 = (int)(P.plane_ld >> 1), nw2 = (P.N + 63) >> 6;
        const long long vstride = (long long)P.nplanes * ld2;
        const uint2* planes = reinterpret_cast<const uint2*>(P.planes);
        E.xp = planes + E.vx * vstride;
        E.yp = planes + E.vy * vstride;
        const int nxy = lx < E.rx && ly < E.ry ? pair_count(E.gram, E.ld, E.vx, E.ox, lx, E.vy, E.oy, ly) : 0;
        const unsigned long long cells2 = (unsigned long long)((E.rx - 1) * (E.ry - 1)) * (unsigned)((P.N + 31) >> 5);
        bool done = false;
        for (int rb = r0; rb < r1 && !done; rb += 32) {
            // the conditioning variables of the next 32 ranks, one per lane
            int v = 0, rz = 0, oz = 0;
            const int rk = rb + lane;
            if (rk < r1) {
                const bool xside = rk < w.cnt_i;
                const int t = xside ? rk : rk - (int)w.cnt_i;
                v = P.nbr[(long long)(xside ? w.i : w.j) * P.n + (t < (xside ? w.posj : w.posi) ? t : t + 1)];
                rz = P.ar[v];
                oz = P.off[v];
            }
            const int m = min(32, r1 - rb);
            for (int q = 0; q < m; ++q) {
                if (!whole && q > 0) {
                    unsigned long long ma = 0;
                    if (lane == 0) ma = *((volatile unsigned long long*)min_accept);
                    if (LOOP && lane == 0) atomicAdd(&a.ctr->beat, 1u);
                    if ((unsigned long long)(rb + q) > __shfl_sync(0xffffffffu, ma, 0)) {
                        done = true;
                        break;
                    }
                }
                const int vz = __shfl_sync(0xffffffffu, v, q), rzq = __shfl_sync(0xffffffffu, rz, q);
                const int dec = marg_test(a, P, E, vz, rzq, __shfl_sync(0xffffffffu, oz, q), nxy, lx, ly, ld2, nw2,
                                          s_cells[threadIdx.x >> 5]);
                tests += 1;
                work += cells2 * (unsigned)(rzq - 1);
                if (dec) {
                    if (lane == 0) atomicMin(min_accept, (unsigned long long)(rb + q));
                    done = true;
                    break;
                }
            }
        }
    }
    if (lane == 0 && tests) {
        atomicAdd(&a.ctr->tests, tests);
        atomicAdd(&a.ctr->popc_work, work);
    }
}

// --------------------------------------------------------------------------
// Depth 0 of small problems: every pair's table by POPC into the Gram (upper
// triangle and the diagonal of each diagonal block), and the pair's decision.
// One warp per pair, a vertex's pairs side by side.  (The tensor-core Gram
// takes over from 512 one-hot rows and 4,096 samples: its fixed cost, one-hot
// rows, tiles and a separate decision, is about 40 us.)
namespace {

template <int A, int B>
__device__ __forceinline__ void pair_cells(const uint2* __restrict__ x, const uint2* __restrict__ y, int ld2, int nw2,
                                           int N, int lx, int ly, int& n, int& nx, int& ny)
{
    const int lane = threadIdx.x & 31;
    unsigned acc[A][B], ax[A], ay[B];
#pragma unroll
    for (int a = 0; a < A; ++a) {
        ax[a] = 0u;
#pragma unroll
        for (int b = 0; b < B; ++b) acc[a][b] = 0u;
    }
#pragma unroll
    for (int b = 0; b < B; ++b) ay[b] = 0u;
#pragma unroll 1
    for (int w = lane; w < nw2; w += 32) {
        uint2 X[A], Y[B];
#pragma unroll
        for (int a = 0; a < A; ++a) X[a] = __ldg(x + a * ld2 + w);
#pragma unroll
        for (int b = 0; b < B; ++b) Y[b] = __ldg(y + b * ld2 + w);
#pragma unroll
        for (int a = 0; a < A; ++a) {
            ax[a] += __popc(X[a].x) + __popc(X[a].y);
#pragma unroll
            for (int b = 0; b < B; ++b) acc[a][b] += __popc(X[a].x & Y[b].x) + __popc(X[a].y & Y[b].y);
        }
#pragma unroll
        for (int b = 0; b < B; ++b) ay[b] += __popc(Y[b].x) + __popc(Y[b].y);
    }
    int s = 0, tx = 0, ty = 0;   // tx, ty: samples of this lane's value (value 0: -(all others))
#pragma unroll
    for (int a = 0; a < A; ++a) {
        int u = 0;
#pragma unroll
        for (int b = 0; b < B; ++b) u += ie_sign(ly, b) * (int)__reduce_add_sync(0xffffffffu, acc[a][b]);
        s += ie_sign(lx, a) * u;
        tx += ie_sign(lx, a) * (int)__reduce_add_sync(0xffffffffu, ax[a]);
    }
#pragma unroll
    for (int b = 0; b < B; ++b) ty += ie_sign(ly, b) * (int)__reduce_add_sync(0xffffffffu, ay[b]);
    nx = lx == 0 ? N + tx : tx;
    ny = ly == 0 ? N + ty : ty;
    n = s + (lx > 0 ? (ly > 0 ? 0 : nx) : (ly > 0 ? ny : nx + ny - N));
}

// The pair's decision in exact FP64 (see marg_exact).
__device__ __noinline__ int pair_exact(const PoolArgs& a, bool cell, int n, int nx, int ny, int N, int df)
{
    double st = 0.0;
    if (cell) {
        const long long p = (long long)n * N, q = (long long)nx * ny;
        if (a.stat == kStatX2) {
            if (q > 0) {
                const double dd = (double)(p - q);
                st = dd * dd / ((double)N * (double)nx * (double)ny);
            }
        } else if (n > 0) {
            st = 2.0 * (double)n * log1p((double)(p - q) / (double)q);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) st += __shfl_xor_sync(0xffffffffu, st, o);
    int dec = 0;
    if ((threadIdx.x & 31) == 0) dec = st < crit_get(a.crit, df, a.alpha, &a.ctr->status);
    return __shfl_sync(0xffffffffu, dec, 0);
}

}  // namespace

template <bool LOOP>
__device__ __forceinline__ void pairs_popc_body(const ProblemDev* probs, const int32_t* vtx_prob,
                                                const int32_t* vtx_first, int total_vertices, int max_n,
                                                const uint8_t* owned, const PoolArgs& a)
{
    DepthCounters* ctr = a.ctr;
    if (blockIdx.x == 0 && threadIdx.x == 0)
        if (DepthRecord* r = depth_rec(ctr, ctr->d)) r->t_tests = gtime();
    const int lane = threadIdx.x & 31, lx = lane / kMA, ly = lane - lx * kMA;
    const long long tasks = (long long)total_vertices * max_n;
    const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
    unsigned long long tests = 0, work = 0;
    for (long long t = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < tasks; t += warps) {
        const int g = (int)(t / max_n), j = (int)(t - (long long)g * max_n);
        const ProblemDev& P = probs[vtx_prob[g]];
        const int i = g - vtx_first[vtx_prob[g]];
        if (j <= i || j >= P.n) continue;
        const int ri = P.ar[i], rj = P.ar[j];
        const int vx = ri >= rj ? i : j, vy = ri >= rj ? j : i;
        const int rx = max(ri, rj), ry = min(ri, rj);
        const int ld2 = (int)(P.plane_ld >> 1), nw2 = (P.N + 63) >> 6;
        const uint2* planes = reinterpret_cast<const uint2*>(P.planes);
        const uint2* x = planes + (long long)vx * P.nplanes * ld2;
        const uint2* y = planes + (long long)vy * P.nplanes * ld2;
        int n = 0, nx = 0, ny = 0;
        switch ((rx - 1) * 4 + ry - 1) {
#define FBN_PAIR(p, q) case (p) * 4 + (q): pair_cells<p, q>(x, y, ld2, nw2, P.N, lx, ly, n, nx, ny); break
            FBN_PAIR(1, 1); FBN_PAIR(2, 1); FBN_PAIR(2, 2); FBN_PAIR(3, 1); FBN_PAIR(3, 2);
            FBN_PAIR(3, 3); FBN_PAIR(4, 1); FBN_PAIR(4, 2); FBN_PAIR(4, 3); FBN_PAIR(4, 4);
#undef FBN_PAIR
            default: break;
        }
        const bool cell = lx < rx && ly < ry;
        const long long ld = P.gram_ld;
        const int ox = P.off[vx], oy = P.off[vy];
        int32_t* G = P.gram;
        if (cell) G[vx < vy ? (ox + lx) * ld + oy + ly : (oy + ly) * ld + ox + lx] = n;
        if (j == i + 1) {   // the single counts of i (and of the last variable)
            const bool ix = vx == i;
            if ((ix ? ly : lx) == 0 && (ix ? lx < rx : ly < ry)) {
                const int o = (ix ? ox + lx : oy + ly);
                G[o * (ld + 1)] = ix ? nx : ny;
            }
            if (j == P.n - 1 && (ix ? lx : ly) == 0 && (ix ? ly < ry : lx < rx)) {
                const int o = (ix ? oy + ly : ox + lx);
                G[o * (ld + 1)] = ix ? ny : nx;
            }
        }
        if (owned && !owned[(long long)i * P.n + j]) continue;   // another process tests the pair
        tests += 1;
        if (LOOP && lane == 0 && t >= warps) atomicAdd(&ctr->beat, 1u);
        work += (unsigned long long)((rx - 1) * (ry - 1)) * (unsigned)((P.N + 31) >> 5);
        // the decision: one stratum holding every sample
        float acc = 0.0f, mag = 0.0f;
        if (cell && nx > 0 && ny > 0) marg_term(n, P.N, nx, ny, P.N < 65536, a.stat, acc, mag);
        int df = (rx - 1) * (ry - 1);
        if (a.df_mode) {
            const int qx = __popc(__ballot_sync(0xffffffffu, cell && ly == 0 && nx > 0));
            const int qy = __popc(__ballot_sync(0xffffffffu, cell && lx == 0 && ny > 0));
            df = (qx - 1) * (qy - 1);
        }
        int dec = 1;
        if (df > 0) {
            float2 cr = make_float2(0.0f, 0.0f);
            if (lane == 0) cr = a.crit.dense_f[df];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                acc += __shfl_xor_sync(0xffffffffu, acc, o);
                mag += __shfl_xor_sync(0xffffffffu, mag, o);
            }
            dec = -1;
            if (cr.y > 0.0f) dec = decide_from_sums(acc, mag, 1.0f, 5.0f, a.stat, cr.x, cr.y, kMargTermRel);
            dec = __shfl_sync(0xffffffffu, dec, 0);
            if (dec < 0) dec = pair_exact(a, cell, n, nx, ny, P.N, df);
        }
        // the complete graph's snapshot: j is entry j - 1 of i's list
        if (dec && lane == 0) a.min_accept[P.eid[(long long)i * P.n + j - 1]] = 0;
    }
    if (lane == 0 && tests) {
        atomicAdd(&ctr->tests, tests);
        atomicAdd(&ctr->popc_work, work);
    }
}

}  // namespace fbn
