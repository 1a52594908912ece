// fbn_device.cuh -- group-level conditional-independence test for sm_103a:
// contingency counts over all samples, marginals, G^2 and the decision
// against alpha, plus the lexicographic unranking of conditioning sets.
//
// A "group" is the set of threads that runs one test: one warp (G = 32) or a
// whole CTA (G = kTestThreads).  Warp groups let many small tests run
// concurrently on an SM so that the latency of one test's setup and epilogue
// is hidden by the others; CTA groups serve tables too big for a warp's share
// of shared memory.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "fbn_internal.cuh"

namespace fbn {

// --------------------------------------------------------------------------
// Chi-square survival function Q(df/2, g2/2) in FP64, integer df.
// Series for the lower regularised gamma P (Abramowitz & Stegun 6.5.29) when
// x < a + 1; else, up to df 64, the finite sum from its largest term down
// (A&S 26.4.4, 26.4.5: 16 terms on average, four independent quotients at a
// time), and above that the continued fraction (A&S 6.5.31) by the modified
// Lentz method (13 to 22 steps of two dependent divisions, where the sum grows to
// 48 terms at df 400 and 185 in the thousands).  First depth 0 of 101 variables,
// a new alpha: 0.58 ms with the fraction alone, 0.19 with the sum up to df 64 or
// 256.  Against 40 digits both are off by what lgamma and exp leave: 3.4e-15 on
// average up to df 60, 5.3e-14 up to 400.
// lgamma/log/exp are CUDA's.  An iteration cap sets kStatusNumeric in *status
// (and *capped when given).
// lg: ln Gamma(df / 2); *pref receives x^a e^-x / Gamma(a) with a = df / 2, x = g2 / 2.
static __device__ __noinline__ double chisq_q(double df, double g2, double lg, double* pref, unsigned* status,
                                              bool* capped = nullptr)
{
    *pref = 0.0;
    if (!(g2 > 0.0)) return 1.0;
    const double a = 0.5 * df, x = 0.5 * g2;
    const double log_pref = a * log(x) - x - lg;
    *pref = exp(log_pref);
    const int kMaxIt = 1 << 20;
    const double kEps = 5e-16, kTiny = 1e-300;
    if (x < a + 1.0) {
        double term = 1.0 / a, sum = term, den = a;
        int it = 0;
        for (; it < kMaxIt && !(term < sum * kEps); ++it) {
            double t[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                den += 1.0;
                t[k] = x / den;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                term *= t[k];
                sum += term;
            }
        }
        if (it == kMaxIt) {
            atomicOr(status, kStatusNumeric);
            if (capped) *capped = true;
        }
        const double q = 1.0 - sum * *pref;
        return q < 0.0 ? 0.0 : q;
    }
    double q;
    int it = 0;
    if (df <= 64.0) {
        double term = a < 1.0 ? 0.0 : 1.0, sum = term, left = a;
        for (; term > sum * kEps; ++it) {   // at most 8 rounds
            double t[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                left -= 1.0;
                t[k] = left < 1.0 ? 0.0 : left / x;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                term *= t[k];
                sum += term;
            }
        }
        q = sum * (*pref / x) + (fmod(df, 2.0) != 0.0 ? erfc(sqrt(x)) : 0.0);
    } else {
        double b = x + 1.0 - a, c = 1.0 / kTiny, d = 1.0 / b, h = d;
        for (it = 1; it < kMaxIt; ++it) {
            const double an = -(double)it * ((double)it - a);
            b += 2.0;
            d = an * d + b;
            if (fabs(d) < kTiny) d = kTiny;
            c = b + an / c;
            if (fabs(c) < kTiny) c = kTiny;
            d = 1.0 / d;
            const double del = d * c;
            h *= del;
            if (fabs(del - 1.0) < kEps) break;
        }
        if (it == kMaxIt) {
            atomicOr(status, kStatusNumeric);
            if (capped) *capped = true;
        }
        q = *pref * h;
    }
    return q > 1.0 ? 1.0 : q;
}

// Critical value of the test: the G^2 at which Q(df/2, G^2/2) = alpha.  Q is
// strictly decreasing in G^2, so "p > alpha" is exactly "G^2 < crit".  Found
// by a safeguarded Newton iteration on ln Q (slope -pref / (G^2 Q); nearly linear
// in the tail) inside a bracket [lo, hi] with Q(lo) > alpha >= Q(hi).  It starts
// from the Wilson-Hilferty cube (A&S 26.4.17) with the normal quantile of A&S
// 26.2.23 and ends with the first step below 1e-10 of G^2, whose error is that
// step's square: 3 evaluations of Q, where Newton on Q from the middle of a wide
// bracket, down to a step of 1e-15, took 17 to 22 (steps at the rounding of Q fell
// outside the bracket and were bisected), each a serial chain of FP64 divisions
// that a first call runs for every new df in every group that meets it.  Against 30
// digits the values of df 1 to 400 are off by 6.4e-16 on average over five alphas,
// before and now.  First pass of new handles: 256 problems 34.8 -> 17.9 ms, 20
// variables 3.7 -> 0.9, 101 with the observed df 10.2 -> 2.4.
static __device__ __noinline__ double chisq_crit(double df, double alpha, unsigned* status, bool* capped = nullptr)
{
    const double a = 0.5 * df, lg = lgamma(a);
    const double t = sqrt(-2.0 * log(fmin(alpha, 1.0 - alpha)));
    double z = t - (2.515517 + t * (0.802853 + t * 0.010328)) / (1.0 + t * (1.432788 + t * (0.189269 + t * 0.001308)));
    if (alpha > 0.5) z = -z;
    const double h = 2.0 / (9.0 * df), c = 1.0 - h + z * sqrt(h);
    double lo = 0.0, hi = INFINITY, x = df * c * c * c;
    if (!(x > 1e-3 * df)) x = 0.5 * df;   // far in the lower tail
    for (int it = 0; it < 200; ++it) {
        double pref;
        const double q = chisq_q(df, x, lg, &pref, status, capped);
        if (q > alpha) lo = x; else hi = x;
        // Newton on ln Q, whose slope is -pref / (G^2 Q); the last step's error is its square
        const double ln = q > 0.5 * alpha && q < 2.0 * alpha ? log1p((q - alpha) / alpha) : log(q / alpha);
        const double step = q > 0.0 && pref > 0.0 ? ln * q * x / pref : NAN;
        if (fabs(step) <= 1e-10 * x) return x + step;
        double nx = x + step;
        if (!(nx > lo && nx < hi)) nx = hi < INFINITY ? 0.5 * (lo + hi) : 2.0 * x;
        if (hi - lo <= 1e-15 * lo) return nx;
        x = nx;
    }
    return x;
}

// Critical values for one alpha.  Small df: a dense table whose slot holds 0
// until a test computes the value and stores it (the value is its own
// payload: a reader sees 0 or the value, and one that sees 0 computes it
// too; a value whose computation hit an iteration cap is never stored).
// Larger df: an open-addressing cache keyed by df; a slot is claimed with a
// CAS to -1, filled, then published with a release store of the key; readers
// that see -1 compute the value themselves.  No thread waits on another.
using CritTable = CritTableDev;

__device__ __forceinline__ long long ld_acquire(const long long* p)
{
    long long v;
    asm volatile("ld.acquire.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release(long long* p, long long v)
{
    asm volatile("st.release.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ double crit_get(const CritTable& t, long long df, double alpha, unsigned* status)
{
    if (df < t.dense_n) {
        const double v = t.dense[df];
        if (v > 0.0) return v;
        bool capped = false;
        const double c = chisq_crit((double)df, alpha, status, &capped);
        if (!capped) {
            t.dense[df] = c;
            if (t.dense_f) t.dense_f[df] = make_float2(__double2float_rd(c), __double2float_ru(c));
            if (t.dense_q) t.dense_q[df] = (long long)floor(c * 0.5 * 68719476736.0);   // 2^kLutBits
        }
        return c;
    }
    unsigned h = (unsigned)(df * 0x9E3779B97F4A7C15ULL >> 40) & (unsigned)(t.cap - 1);
    for (int probe = 0; probe < 32; ++probe, h = (h + 1) & (unsigned)(t.cap - 1)) {
        const long long k = ld_acquire(t.keys + h);
        if (k == df) return t.vals[h];
        if (k == 0) {
            const double c = chisq_crit((double)df, alpha, status);
            if (atomicCAS((unsigned long long*)(t.keys + h), 0ULL, (unsigned long long)-1LL) == 0ULL) {
                t.vals[h] = c;
                st_release(t.keys + h, df);
            }
            return c;
        }
        if (k == -1) return chisq_crit((double)df, alpha, status);
    }
    return chisq_crit((double)df, alpha, status);
}

// --------------------------------------------------------------------------
// Conditioning sets on the fly (Section IV-C): the r-th q-subset of {0..p-1}
// in lexicographic order, from a table of binomials B[n][k] = C(n, k).
__device__ __forceinline__ long long binom_at(const long long* B, int n, int k)
{
    if (k < 0 || n < k) return 0;
    return __ldg(B + (long long)n * kBinomCols + k);
}

__device__ __forceinline__ void unrank_lex(long long r, int p, int q, const long long* B, int* out)
{
    int c = 0;
    for (int k = 0; k < q; ++k) {
        if (k == q - 1) {            // last position: one subset per candidate
            out[k] = c + (int)r;
            return;
        }
        for (;;) {
            const long long cnt = binom_at(B, p - c - 1, q - k - 1);
            if (r < cnt) break;
            r -= cnt;
            ++c;
        }
        out[k] = c++;
    }
}

// Next q-subset of {0..p-1} in lexicographic order; false after the last.
__device__ __forceinline__ bool next_subset(int p, int q, int* c)
{
    int k = q - 1;
    while (k >= 0 && c[k] == p - q + k) --k;
    if (k < 0) return false;
    c[k] += 1;
    for (int l = k + 1; l < q; ++l) c[l] = c[l - 1] + 1;
    return true;
}

// --------------------------------------------------------------------------
// One CI test as seen by its group, in shared memory.
// rows = [S_0 .. S_{d-1}, X, Y]; the cell of a sample is the mixed-radix
// number of its values in that order: ((z * r_x + x) * r_y + y).
struct TestSpec {
    const uint8_t* rows[kMaxRows];
    int rad[kMaxRows];
    int nrows;        // d + 2
    int rx, ry;
    int N;
    long long cells;  // product of all radices
};

template <int G>
struct Grp {
    static_assert(G == 32 || G == 64 || G == 128 || G == kTestThreads || G == kBigThreads, "group size");
    static constexpr int kWarps = G / 32;
    static __device__ __forceinline__ int rank() { return (int)(threadIdx.x % G); }
    static __device__ __forceinline__ int gid() { return (int)(threadIdx.x / G); }
    static __device__ __forceinline__ void sync()
    {
        if (G == 32) {
            __syncwarp();
        } else if (G >= kTestThreads) {   // the whole CTA
            __syncthreads();
        } else {   // named barrier 1 + group index, G threads
            asm volatile("bar.sync %0, %1;" ::"r"(1 + gid()), "r"(G) : "memory");
        }
    }
};

// Sum over the group; every thread of the group gets the total.  red: the
// CTA's scratch of 32 entries of 8 bytes, of which the group uses kWarps.
template <int G, typename T>
__device__ __forceinline__ T grp_sum(T v, T* red)
{
    static_assert(sizeof(T) == 8, "a smaller type's slots would overlap another group's");
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (G == 32) return v;
    T* r = red + Grp<G>::gid() * Grp<G>::kWarps;
    Grp<G>::sync();
    if ((threadIdx.x & 31) == 0) r[Grp<G>::rank() >> 5] = v;
    Grp<G>::sync();
    T t = 0;
#pragma unroll
    for (int w = 0; w < Grp<G>::kWarps; ++w) t += r[w];
    return t;
}

// --------------------------------------------------------------------------
// Counting: one loop for every table in shared memory.  A table of C cells is
// kept in K interleaved copies (K a power of two, at most 32):
// copy k of cell c is word c K + k, and thread t counts into copy t mod K.  K is
// the largest up to 32 that fits, so small tables get a copy per lane (no two
// threads of a warp meet in a word or a bank) and large ones at least a few: a warp's
// 32 updates of one shared copy met 3.9 deep in a cell (depth 2, arities 2-4),
// in 4 copies 2.2, in 8 copies 1.8.  The update is a shared-memory reduction,
// so consecutive samples do not wait on each other.  One loop with a runtime
// copy count instead of one per strategy keeps the pool's code small: every
// test runs through all of it, and instruction fetch was a third of the
// histogram pools' stalls.
struct SharedCounter {
    unsigned base;   // shared address of this thread's copy of cell 0
    unsigned step;   // bytes from a cell to the next: 4 K
    __device__ __forceinline__ void bump(unsigned idx) const
    {
        asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(base + idx * step) : "memory");
    }
};

struct GlobalCounter {
    int* base;
    __device__ __forceinline__ void bump(unsigned idx) const { atomicAdd(base + idx, 1); }
};

// The ragged tail: samples past the last whole 16-sample vector.
template <class Counter>
__device__ __forceinline__ void count_tail(const TestSpec& s, const Counter& cnt, int rank, int G)
{
    for (int t = (s.N & ~15) + rank; t < s.N; t += G) {
        unsigned idx = s.rows[0][t];
        for (int k = 1; k < s.nrows; ++k) idx = idx * (unsigned)s.rad[k] + s.rows[k][t];
        cnt.bump(idx);
    }
}

// Tables of at most 256 cells: every partial index of a sample fits one byte,
// so the four samples of a 32-bit word advance together in its four bytes --
// acc * r_k + row_k never carries out of a byte because the result stays below
// the cells counted so far.  One IMAD per row and 4 samples, then one byte
// extraction per sample.  The next kCountDepth vectors of each row are in
// flight while one is counted.
// (measured at depth 2 of 256 problems: 1 vector ahead 2.9 ms at three CTAs per
// SM and 3.1 at two; 2 ahead at two CTAs 2.3; 3 ahead 2.1 there, the others
// unchanged, for 32 more registers)
constexpr int kCountDepth = 2;
template <int NR>
__device__ __forceinline__ void count_bytes(const TestSpec& s, const SharedCounter& cnt, int rank, int G)
{
    const int nvec = s.N >> 4;
    const uint4* r[NR];
    unsigned rad[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        r[k] = reinterpret_cast<const uint4*>(s.rows[k]);
        rad[k] = (unsigned)s.rad[k];
    }
    uint4 w[kCountDepth][NR];
    const int last = nvec - 1;
    if (rank > last) return;
#pragma unroll
    for (int i = 0; i < kCountDepth; ++i)
#pragma unroll
        for (int k = 0; k < NR; ++k) w[i][k] = __ldg(r[k] + min(rank + i * G, last));
#pragma unroll 1
    for (int v = rank; v <= last; v += kCountDepth * G) {
#pragma unroll
        for (int i = 0; i < kCountDepth; ++i) {
            if (i && v + i * G > last) break;
            uint4 a = w[i][0];
#pragma unroll
            for (int k = 1; k < NR; ++k) {
                a.x = a.x * rad[k] + w[i][k].x; a.y = a.y * rad[k] + w[i][k].y;
                a.z = a.z * rad[k] + w[i][k].z; a.w = a.w * rad[k] + w[i][k].w;
            }
            const int vn = min(v + (kCountDepth + i) * G, last);
#pragma unroll
            for (int k = 0; k < NR; ++k) w[i][k] = __ldg(r[k] + vn);
            const unsigned q[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                cnt.bump(__byte_perm(q[t], 0u, 0x4440));
                cnt.bump(__byte_perm(q[t], 0u, 0x4441));
                cnt.bump(__byte_perm(q[t], 0u, 0x4442));
                cnt.bump(__byte_perm(q[t], 0u, 0x4443));
            }
        }
    }
}

// At most 65,536 cells: the indices of two samples ride in the 16-bit halves of
// one register (every partial index is below the cells), one IMAD for both.
// NR = 0: any number of rows.
template <int NR, class Counter>
__device__ __forceinline__ void count_packed(const TestSpec& s, const Counter& cnt, int rank, int G)
{
    const int nvec = s.N >> 4;
    const int nr = NR > 0 ? NR : s.nrows;
    constexpr int kBuf = NR > 0 ? NR : 1;
    uint4 w[kBuf];
    const int last = nvec - 1;
    if (NR > 0 && rank <= last) {
#pragma unroll
        for (int k = 0; k < kBuf; ++k) w[k] = __ldg(reinterpret_cast<const uint4*>(s.rows[k]) + rank);
    }
#pragma unroll 1
    for (int v = rank; v <= last; v += G) {
        unsigned acc[8];
        if (NR > 0) {
#pragma unroll
            for (int k = 0; k < kBuf; ++k) {
                const unsigned ws[4] = {w[k].x, w[k].y, w[k].z, w[k].w};
                const unsigned rk = (unsigned)s.rad[k];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const unsigned lo = __byte_perm(ws[q], 0u, 0x4140), hi = __byte_perm(ws[q], 0u, 0x4342);
                    acc[2 * q] = k ? acc[2 * q] * rk + lo : lo;          // bytes 0, 1 -> halves
                    acc[2 * q + 1] = k ? acc[2 * q + 1] * rk + hi : hi;  // bytes 2, 3 -> halves
                }
            }
            const int vn = min(v + G, last);
#pragma unroll
            for (int k = 0; k < kBuf; ++k) w[k] = __ldg(reinterpret_cast<const uint4*>(s.rows[k]) + vn);
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) acc[q] = 0u;
            for (int k = 0; k < nr; ++k) {
                const uint4 x = __ldg(reinterpret_cast<const uint4*>(s.rows[k]) + v);
                const unsigned ws[4] = {x.x, x.y, x.z, x.w};
                const unsigned rk = (unsigned)s.rad[k];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    acc[2 * q] = acc[2 * q] * rk + __byte_perm(ws[q], 0u, 0x4140);
                    acc[2 * q + 1] = acc[2 * q + 1] * rk + __byte_perm(ws[q], 0u, 0x4342);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            cnt.bump(acc[q] & 0xFFFFu);
            cnt.bump(acc[q] >> 16);
        }
    }
}

// Above: one sample per 32-bit index.
template <class Counter>
__device__ __forceinline__ void count_wide(const TestSpec& s, const Counter& cnt, int rank, int G)
{
    const int nvec = s.N >> 4;
#pragma unroll 1
    for (int v = rank; v < nvec; v += G) {
        unsigned idx[16];
#pragma unroll
        for (int b = 0; b < 16; ++b) idx[b] = 0u;
        for (int k = 0; k < s.nrows; ++k) {
            const uint4 w = __ldg(reinterpret_cast<const uint4*>(s.rows[k]) + v);
            const unsigned rk = (unsigned)s.rad[k];
            const unsigned ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int b = 0; b < 16; ++b) idx[b] = idx[b] * rk + ((ws[b >> 2] >> ((b & 3) * 8)) & 0xFFu);
        }
#pragma unroll
        for (int b = 0; b < 16; ++b) cnt.bump(idx[b]);
    }
}

// The samples of the test into shared copies, by thread `rank` of G.
static __device__ __noinline__ void count_shared(const TestSpec& s, SharedCounter cnt, int rank, int G)
{
    if (s.cells <= 256) {
        switch (s.nrows) {
            case 2: count_bytes<2>(s, cnt, rank, G); break;
            case 3: count_bytes<3>(s, cnt, rank, G); break;
            case 4: count_bytes<4>(s, cnt, rank, G); break;
            case 5: count_bytes<5>(s, cnt, rank, G); break;
            default: count_packed<0>(s, cnt, rank, G); break;
        }
    } else {
        switch (s.nrows) {
            case 2: count_packed<2>(s, cnt, rank, G); break;
            case 3: count_packed<3>(s, cnt, rank, G); break;
            case 4: count_packed<4>(s, cnt, rank, G); break;
            case 5: count_packed<5>(s, cnt, rank, G); break;
            default: count_packed<0>(s, cnt, rank, G); break;
        }
    }
    count_tail(s, cnt, rank, G);
}

// The same into one global table.
static __device__ __noinline__ void count_global(const TestSpec& s, int* table, int rank, int G)
{
    const GlobalCounter cnt{table};
    if (s.cells > 65536) count_wide(s, cnt, rank, G);
    else count_packed<0>(s, cnt, rank, G);
    count_tail(s, cnt, rank, G);
}

// Copies of a table of C cells: the most that fit, while zeroing and folding
// them (C K words each) stays below the samples counted, and at most one per lane of
// a warp (with one per thread of a CTA few threads fold many words each: the
// edge-level form of 300 variables x 30,000 samples 3.72 ms, 3.40 with 32); where the marginals are
// kept too, one from kOneCopy cells on, where a warp's updates hardly meet (13 M
// tests of 7,776 cells and 50,000 samples, X^2 with the observed df: 1,357 ms with
// two copies, 1,230 with one; G^2 from the n ln n table: 637 and 639).
constexpr long long kOneCopy = 4096;
template <int G>
__device__ __forceinline__ int table_copies(long long C, long long slice_ints, int N, bool need_marg)
{
    int K = need_marg && C >= kOneCopy ? 1 : 32;
    while (K > 1 && (C * K > slice_ints || 2 * C * K > N)) K >>= 1;
    return K;
}

// Count the table of the test.  Returns the table T -- in the slice, or in the
// global scratch when the slice cannot hold it (with its marginals when the
// caller needs them: need_marg) -- and sets *M to the space for the marginals;
// nullptr when the table fits neither.
template <int G>
__device__ __forceinline__ int* grp_table(const TestSpec& s, int* slice, long long slice_ints, int* gtab,
                                          long long gtab_ints, bool need_marg, int** M)
{
    const int C = (int)s.cells;   // <= kMaxCells
    const long long marg = need_marg ? (long long)(C / (s.rx * s.ry)) * (s.rx + s.ry + 1) : 0;
    const int r = Grp<G>::rank(), lane = threadIdx.x & 31;
    if (C + marg > slice_ints) {
        if (gtab == nullptr || C + marg > gtab_ints) return nullptr;
        for (int k = r; k < C; k += G) gtab[k] = 0;
        Grp<G>::sync();
        count_global(s, gtab, r, G);
        Grp<G>::sync();
        *M = marg <= slice_ints ? slice : gtab + C;
        return gtab;
    }
    const int K = table_copies<G>(C, slice_ints, s.N, need_marg);
    uint4* z = reinterpret_cast<uint4*>(slice);   // slices are whole 16-byte words
    for (int k = r; k < (C * K + 3) / 4; k += G) z[k] = make_uint4(0u, 0u, 0u, 0u);
    Grp<G>::sync();
    SharedCounter cnt;
    cnt.base = (unsigned)__cvta_generic_to_shared(slice) + 4u * (unsigned)(r & (K - 1));
    cnt.step = 4u * (unsigned)K;
    count_shared(s, cnt, r, G);
    Grp<G>::sync();
    if (K > 1) {
        // fold in place: cell c's sum goes to word c, which lies in copies read
        // in this round or before (words past them are not written); lanes
        // start at rotated words of their cells (no bank conflicts)
        const int rot = K >= 32 ? lane : (lane * K) >> 5;
        for (int c0 = 0; c0 < C; c0 += G) {
            const int c = c0 + r;
            int sum = 0;
            if (c < C) {
                if (K == 2) {
                    const int2 v = reinterpret_cast<const int2*>(slice)[c];
                    sum = v.x + v.y;
                } else {
                    const int4* row = reinterpret_cast<const int4*>(slice + (long long)c * K);
#pragma unroll 2
                    for (int q = 0; q < K / 4; ++q) {
                        const int4 v = row[(q + rot) & (K / 4 - 1)];
                        sum += v.x + v.y + v.z + v.w;
                    }
                }
            }
            Grp<G>::sync();
            if (c < C) slice[c] = sum;
        }
        Grp<G>::sync();
    }
    *M = slice + C;
    return slice;
}

// c / d for c, d < 2^16 as one multiplication (the general division is some 25
// instructions, of which a cell of a decision took two).
struct Divider {
    unsigned m, d;
    bool small;   // every dividend is below 2^16
    __device__ __forceinline__ Divider(int divisor, int dividends)
        : m(divisor == 1 ? 0u : 0xFFFFFFFFu / (unsigned)divisor + 1u), d((unsigned)divisor), small(dividends <= 65536)
    {
    }
    __device__ __forceinline__ int operator()(int c) const   // m = ceil(2^32 / d): exact while c d < 2^32
    {
        return m == 0 ? c : small ? (int)__umulhi((unsigned)c, m) : c / (int)d;
    }
};

// Marginals N_x+z [nz*rx], N_+yz [nz*ry], N_++z [nz] into M.
template <int G>
__device__ __forceinline__ void grp_marginals(const TestSpec& s, const int* T, int* M)
{
    // cells <= kMaxCells < 2^31: 32-bit indices throughout
    const int rx = s.rx, ry = s.ry;
    const int nz = (int)s.cells / (rx * ry);
    int* Nxz = M;
    int* Nyz = M + nz * rx;
    int* Nzz = Nyz + nz * ry;
    const int r = Grp<G>::rank();
    for (int k = r; k < nz * rx; k += G) {
        int sum = 0;
        for (int y = 0; y < ry; ++y) sum += T[k * ry + y];
        Nxz[k] = sum;
    }
    const Divider by_ry(ry, nz * ry);
    for (int k = r; k < nz * ry; k += G) {
        const int z = by_ry(k);
        const int y = k - z * ry;
        int sum = 0;
        for (int x = 0; x < rx; ++x) sum += T[(z * rx + x) * ry + y];
        Nyz[k] = sum;
    }
    Grp<G>::sync();
    for (int z = r; z < nz; z += G) {
        int sum = 0;
        for (int x = 0; x < rx; ++x) sum += Nxz[z * rx + x];
        Nzz[z] = sum;
    }
    Grp<G>::sync();
}

// Exact G^2 = 2 sum N ln(N / E) in FP64 (every thread of the group gets it).
// The ratio N / E = (N_xyz N_++z) / (N_x+z N_+yz) is formed in exact 64-bit
// integers and its log taken as log1p of the exact difference over the
// denominator.
template <int G>
__device__ __forceinline__ double grp_g2_exact(const TestSpec& s, const int* T, const int* M, double* red)
{
    const int rx = s.rx, ry = s.ry, rxy = rx * ry, C = (int)s.cells;
    const int nz = C / rxy;
    const int* Nxz = M;
    const int* Nyz = M + nz * rx;
    const int* Nzz = Nyz + nz * ry;
    double acc = 0.0;
    for (int c = Grp<G>::rank(); c < C; c += G) {
        const int n = T[c];
        if (n == 0) continue;
        const int z = c / rxy;
        const int rem = c - z * rxy;
        const int x = rem / ry, y = rem - x * ry;
        const long long a = (long long)n * Nzz[z];
        const long long b = (long long)Nxz[z * rx + x] * Nyz[z * ry + y];
        acc += (double)n * log1p((double)(a - b) / (double)b);
    }
    return 2.0 * grp_sum<G>(acc, red);
}

// CI-test statistics: G^2 (Section III-B) or Pearson's X^2 of the same table.
constexpr int kStatG2 = 0;
constexpr int kStatX2 = 1;

// Exact Pearson X^2 = sum (N - E)^2 / E in FP64 over cells with E > 0 (empty
// cells included), each term (N_xyz N_++z - N_x+z N_+yz)^2 / (N_++z N_x+z
// N_+yz) with the difference an exact 64-bit integer.
template <int G>
__device__ __forceinline__ double grp_x2_exact(const TestSpec& s, const int* T, const int* M, double* red)
{
    const int rx = s.rx, ry = s.ry, rxy = rx * ry, C = (int)s.cells;
    const int nz = C / rxy;
    const int* Nxz = M;
    const int* Nyz = M + nz * rx;
    const int* Nzz = Nyz + nz * ry;
    double acc = 0.0;
    for (int c = Grp<G>::rank(); c < C; c += G) {
        const int n = T[c];
        const int z = c / rxy;
        const int rem = c - z * rxy;
        const int x = rem / ry, y = rem - x * ry;
        const long long nx = Nxz[z * rx + x], ny = Nyz[z * ry + y];
        if (nx == 0 || ny == 0) continue;
        const double dd = (double)((long long)n * Nzz[z] - nx * ny);
        acc += dd * dd / ((double)Nzz[z] * (double)nx * (double)ny);
    }
    return grp_sum<G>(acc, red);
}

// Degrees of freedom of the observed table: sum over strata with N_++z > 0 of
// (values of X with N_x+z > 0 - 1)(values of Y with N_+yz > 0 - 1).
template <int G>
__device__ __forceinline__ long long grp_df_adjusted(const TestSpec& s, const int* M, double* red)
{
    const int rx = s.rx, ry = s.ry;
    const int nz = (int)s.cells / (rx * ry);
    const int* Nxz = M;
    const int* Nyz = M + nz * rx;
    long long acc = 0;   // whole numbers: additions in FP64 take a test of 32 cells a ninth longer
    for (int z = Grp<G>::rank(); z < nz; z += G) {
        int ax = 0, ay = 0;
        for (int x = 0; x < rx; ++x) ax += Nxz[z * rx + x] > 0;
        for (int y = 0; y < ry; ++y) ay += Nyz[z * ry + y] > 0;
        if (ax > 0 && ay > 0) acc += (ax - 1) * (ay - 1);
    }
    return grp_sum<G>(acc, reinterpret_cast<long long*>(red));
}

// One FP32 term of the bounded decisions.  G^2: n ln(N / E) with the ratio
// N / E = (n N_++z) / (N_x+z N_+yz) from exact 64-bit integers, its log taken
// as log1p of the exact difference over the denominator (n > 0).  X^2:
// (n N_++z - N_x+z N_+yz)^2 / (N_++z N_x+z N_+yz) with the difference exact,
// skipped when a margin is empty.
// Below 65,536 samples (narrow) the products fit 32 bits: the same values, without
// 64-bit conversions, which run at the FP64 rate.
__device__ __forceinline__ void product_floats(int n, int nzz, int nx, int ny, bool narrow, float& fa, float& fb, float& fd)
{
    if (narrow) {
        const unsigned a = (unsigned)n * (unsigned)nzz, b = (unsigned)nx * (unsigned)ny;
        fa = (float)a;
        fb = (float)b;
        fd = a >= b ? (float)(a - b) : -(float)(b - a);
    } else {
        const long long a = (long long)n * nzz, b = (long long)nx * ny;
        fa = (float)a;
        fb = (float)b;
        fd = (float)(a - b);
    }
}

__device__ __forceinline__ void g2_term(int n, int nzz, int nx, int ny, bool narrow, float& acc, float& mag)
{
    float fa, fb, fd;
    product_floats(n, nzz, nx, ny, narrow, fa, fb, fd);
    const float delta = fd / fb;
    const float L = fabsf(delta) < 0.5f ? log1pf(delta) : logf(fa / fb);
    const float t = (float)n * L;
    acc += t;
    mag += fabsf(t);
}

__device__ __forceinline__ void x2_term(int n, int nzz, int nx, int ny, bool narrow, float& acc)
{
    if (nx == 0 || ny == 0) return;
    float fa, fb, fd;
    product_floats(n, nzz, nx, ny, narrow, fa, fb, fd);
    acc += fd * fd / ((float)nzz * (float)nx * (float)ny);
}

// The bounded comparison shared by the FP32 decisions: sum = the group's FP32
// sum of the terms, mag = the sum of their magnitudes, per_thread = terms a
// thread added, levels = the additions across threads a value goes through, term_rel
// = a bound of a term's error against its own magnitude.  The
// error analysis is the one stated for grp_decide_bound below.  Returns 1
// (accept), 0 (reject) or -1 (the band straddles the bracket of crit).
__device__ __forceinline__ int decide_from_sums(float sum, float mag, float per_thread, float levels, int stat,
                                                float crit_lo, float crit_hi, float term_rel)
{
    const float rel = __fmul_ru(2.0f, __fadd_ru(term_rel, __fmul_ru(__fadd_ru(per_thread, levels), 6.0e-8f)));
    const float scale = stat == kStatX2 ? 1.0f : 2.0f;   // G^2 = 2 sum; exact scaling
    const float st = scale * sum;
    const float err = __fadd_ru(__fmul_ru(__fmul_ru(__fmul_ru(scale, rel), fabsf(mag)), 1.0001f), 1e-9f);
    if (__fadd_ru(st, err) < crit_lo) return 1;
    if (__fadd_rd(st, -err) >= crit_hi) return 0;
    return -1;
}

// One FP32 term of the bounded decision from a cell and its margins.  Below
// 65,536 samples both products of the ratio fit 32 bits.  G^2: n ln(N / E) with
// the exact difference D = n N_z - N_xz N_yz; ln as 2 atanh(D / (sum of the two
// products)) by its series while the ratio is within [1/2, 2] (|s| <= 1/3: the
// terms left out are below 2e-9 of the sum), else as lg2 of the ratio.  64-bit
// integers are converted by halves (the single conversion runs at the FP64 rate).
// A term's error against itself, at most: in the series D and the sum (1.2e-7 and
// 1.8e-7) and the quotient (2 ulp: 2.4e-7), 1.08 times as much of the logarithm, the
// series and the product with n 2.2e-7: 8.1e-7; past a ratio of 2 two conversions and
// the quotient (4.8e-7 of the ratio, over ln 2), lg2 (2 ulp: 2.4e-7), two products and
// a conversion (1.8e-7): 1.12e-6.  X^2, D^2 / (N_z N_xz N_yz): 7.8e-7.  The largest of
// 2e8 terms measured: 3.6e-7, 5.4e-7 and 4.3e-7.
__device__ __forceinline__ float u64_float(unsigned long long v)   // within 1.2e-7 of itself
{
    return fmaf((float)(unsigned)(v >> 32), 4294967296.0f, (float)(unsigned)v);
}

__device__ __forceinline__ void marg_term(int n, int nz, int nx, int ny, bool narrow, int stat, float& acc, float& mag)
{
    float fd, fa, fb;
    if (narrow) {
        const unsigned p = (unsigned)n * (unsigned)nz, q = (unsigned)nx * (unsigned)ny;
        fd = p >= q ? (float)(p - q) : -(float)(q - p);
        fa = (float)p;
        fb = (float)q;
    } else {
        const unsigned long long p = (unsigned long long)n * (unsigned)nz, q = (unsigned long long)nx * (unsigned)ny;
        fd = p >= q ? u64_float(p - q) : -u64_float(q - p);
        fa = u64_float(p);
        fb = u64_float(q);
    }
    if (stat == kStatX2) {
        if (fb > 0.0f) {
            const float t = __fdividef(fd * fd, fb) / (float)nz;
            acc += t;
            mag += t;
        }
        return;
    }
    const float s = __fdividef(fd, fa + fb);
    const float s2 = s * s;
    float p = 1.0f / 15.0f;
    p = fmaf(p, s2, 1.0f / 13.0f);
    p = fmaf(p, s2, 1.0f / 11.0f);
    p = fmaf(p, s2, 1.0f / 9.0f);
    p = fmaf(p, s2, 1.0f / 7.0f);
    p = fmaf(p, s2, 1.0f / 5.0f);
    p = fmaf(p, s2, 1.0f / 3.0f);
    const float near = 2.0f * fmaf(s * s2, p, s);
    const float far = __log2f(__fdividef(fa, fb)) * 0.693147181f;
    const float t = n > 0 ? (float)n * (fabsf(s) <= 0.33333333f ? near : far) : 0.0f;
    acc += t;
    mag += fabsf(t);
}
constexpr float kMargTermRel = 1.2e-6f;

// Decision "p > alpha" as "G^2 < crit" from FP32 terms under an error bound,
// all in FP32 (the FP64 pipe of this part is 1/64 of FP32, and every thread
// of a group would otherwise run the bound in it).  The terms are evaluated
// with FP32 logarithms -- each within 7e-7 of its own magnitude: the ratio of
// exact integers within 1.8e-7 (two conversions, a quotient), over ln 1.5 at most
// 4.4e-7 of the logarithm, CUDA's logf and log1pf within 1 ulp (1.2e-7), the product
// with n 1.2e-7 -- and summed in FP32: a thread adds at most ceil(C/G) terms, a warp
// its lanes' sums in 5 levels, the group its warps' one after the other, each
// addition erring by at most 6e-8 of the running sum of magnitudes.  G^2 is thus
// within 2 (7e-7 + (ceil(C/G) + 4 + G/32) 6e-8) sum|term| of its exact value; the
// bound is doubled for margin, formed with upward rounding, and compared against a float bracket [lo, hi]
// of crit (lo <= crit <= hi): accept when G^2 + err < lo, reject when G^2 -
// err >= hi (both rounded outward).  Returns 1 (accept), 0 (reject) or -1
// when the band straddles the bracket and the caller decides exactly.
//
// X^2 (stat = kStatX2): each term D^2 / (N_++z N_x+z N_+yz) with D the exact
// integer difference, formed in FP32 within 6e-7 of itself (three conversions,
// a square, two products, a quotient); the terms are non-negative, so the
// running sum of magnitudes is the sum itself, and the same summation bound
// applies without the doubling of G^2.
template <int G>
__device__ __forceinline__ int grp_decide_bound(const TestSpec& s, const int* T, const int* M, float crit_lo,
                                                float crit_hi, double* red, int stat = kStatG2)
{
    const int rx = s.rx, ry = s.ry, rxy = rx * ry, C = (int)s.cells;
    const int nz = C / rxy;
    const int* Nxz = M;
    const int* Nyz = M + nz * rx;
    const int* Nzz = Nyz + nz * ry;
    const Divider by_rxy(rxy, C), by_ry(ry, rxy);
    const bool narrow = s.N < 65536;
    float acc = 0.0f, mag = 0.0f;
    if (stat == kStatX2) {
        for (int c = Grp<G>::rank(); c < C; c += G) {
            const int z = by_rxy(c);
            const int rem = c - z * rxy;
            const int x = by_ry(rem), y = rem - x * ry;
            x2_term(T[c], Nzz[z], Nxz[z * rx + x], Nyz[z * ry + y], narrow, acc);
        }
        mag = acc;
    } else {
        for (int c = Grp<G>::rank(); c < C; c += G) {
            const int n = T[c];
            if (n == 0) continue;
            const int z = by_rxy(c);
            const int rem = c - z * rxy;
            const int x = by_ry(rem), y = rem - x * ry;
            g2_term(n, Nzz[z], Nxz[z * rx + x], Nyz[z * ry + y], narrow, acc, mag);
        }
    }
    float2 v = make_float2(acc, mag);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    if (G > 32) {
        float* r = reinterpret_cast<float*>(red) + Grp<G>::gid() * 2 * Grp<G>::kWarps;
        Grp<G>::sync();
        if ((threadIdx.x & 31) == 0) {
            r[2 * (Grp<G>::rank() >> 5)] = v.x;
            r[2 * (Grp<G>::rank() >> 5) + 1] = v.y;
        }
        Grp<G>::sync();
        v.x = 0.0f;
        v.y = 0.0f;
#pragma unroll
        for (int w = 0; w < Grp<G>::kWarps; ++w) {
            v.x += r[2 * w];
            v.y += r[2 * w + 1];
        }
    }
    const float per_thread = (float)((C + G - 1) / G);   // exact: C < 2^24
    constexpr float levels = 4.0f + (float)Grp<G>::kWarps;
    return decide_from_sums(v.x, v.y, per_thread, levels, stat, crit_lo, crit_hi, stat == kStatX2 ? 6.0e-7f : 7.0e-7f);
}

// --------------------------------------------------------------------------
// G^2 from a table of n ln n.  G^2 / 2 = sum n_xyz ln n_xyz - sum N_x+z ln N_x+z -
// sum N_+yz ln N_+yz + sum N_++z ln N_++z, with n ln n as 64-bit fixed point
// (2^-kLutBits) from a table indexed by the count: the sums are exact, each
// entry within lut_err units of its value, so the comparison with crit needs no
// cell coordinates, logarithms, divisions or marginals per cell, and its error
// (about 1e-7 for 1,000 cells of 50,000 samples) leaves almost no test for the
// FP64 recomputation, where FP32 terms leave about one in 1,000.
constexpr int kLutBits = 36;
constexpr long long kLutMaxN = 1LL << 20;   // 2^20 ln 2^20 < 2^24: 60 bits

// Exact G^2 in FP64 from the table alone (no stored marginals).  Rare.
template <int G>
__device__ __noinline__ double grp_g2_cells(const TestSpec& s, const int* T, double* red)
{
    const int rx = s.rx, ry = s.ry, rxy = rx * ry, C = (int)s.cells;
    double acc = 0.0;
    for (int c = Grp<G>::rank(); c < C; c += G) {
        const int n = T[c];
        if (n == 0) continue;
        const int z = c / rxy, rem = c - z * rxy, x = rem / ry, y = rem - x * ry;
        const int* S = T + z * rxy;
        long long nx = 0, ny = 0, nz = 0;
        for (int q = 0; q < ry; ++q) nx += S[x * ry + q];
        for (int q = 0; q < rx; ++q) ny += S[q * ry + y];
        for (int q = 0; q < rxy; ++q) nz += S[q];
        const long long a = (long long)n * nz, b = nx * ny;
        acc += (double)n * log1p((double)(a - b) / (double)b);
    }
    return 2.0 * grp_sum<G>(acc, red);
}

// Twice this is G^2, in units of 2^-kLutBits (every thread of the group).
template <int G>
__device__ __forceinline__ long long grp_g2_lut(const TestSpec& s, const int* T, const long long* __restrict__ lut,
                                                double* red)
{
    const int rx = s.rx, ry = s.ry, rxy = rx * ry, C = (int)s.cells, r = Grp<G>::rank();
    const int nz = C / rxy;
    long long acc = 0;
#pragma unroll 1
    for (int k = r; k < nz * rx; k += G) {   // rows (x, z): their cells and N_x+z
        int n = 0;
        const int* t = T + k * ry;
#pragma unroll 4
        for (int y = 0; y < ry; ++y) {
            const int v = t[y];
            n += v;
            acc += __ldg(lut + v);
        }
        acc -= __ldg(lut + n);
    }
    const unsigned m = 0xFFFFFFFFu / (unsigned)ry + 1u;   // k / ry = umulhi(k, m) while k ry < 2^32
#pragma unroll 1
    for (int k = r; k < nz * ry; k += G) {   // columns (y, z): N_+yz
        const int z = ry == 1 ? k : (int)__umulhi((unsigned)k, m);
        const int* t = T + z * rxy + (k - z * ry);
        int n = 0;
#pragma unroll 4
        for (int x = 0; x < rx; ++x) n += t[x * ry];
        acc -= __ldg(lut + n);
    }
    // few strata of many cells: a warp each (a reduction costs about 8 cells) instead of
    // a thread each, whose reads rxy apart also meet in a bank when 2 divides rxy often
    // (depth 0 of 40 variables of 100 values x 20,000 samples, one stratum of 10,000
    // cells: 0.30 ms with one thread, 0.05; depth 1 of 40 variables of 8 values x 5,000:
    // 0.47 and 0.42)
    constexpr int W = Grp<G>::kWarps;
    const int meet = max(1, min(nz, 32) * min(rxy & -rxy, 32) / 32);
    if (nz < G && (nz + W - 1) / W * (rxy / 32 + 8) < rxy * meet) {
#pragma unroll 1
        for (int z = r >> 5; z < nz; z += W) {
            int n = 0;
            const int* t = T + z * rxy;
            for (int q = r & 31; q < rxy; q += 32) n += t[q];
            n = __reduce_add_sync(0xffffffffu, n);
            if ((r & 31) == 0) acc += __ldg(lut + n);
        }
    } else {
#pragma unroll 1
        for (int z = r; z < nz; z += G) {    // strata: N_++z
            int n = 0;
            const int* t = T + z * rxy;
#pragma unroll 4
            for (int q = 0; q < rxy; ++q) n += t[q];
            acc += __ldg(lut + n);
        }
    }
    return grp_sum<G>(acc, reinterpret_cast<long long*>(red));
}

}  // namespace fbn
