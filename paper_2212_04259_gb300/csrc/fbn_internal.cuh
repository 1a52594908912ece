// fbn_internal.cuh -- device-side data structures shared by the kernels and the
// host engine of the GB300 PC-stable skeleton library.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace fbn {

constexpr int kMaxD = 30;                 // largest conditioning set supported
constexpr int kMaxRows = kMaxD + 2;       // S rows + X row + Y row
constexpr int kBinomCols = kMaxD + 2;     // binomial table columns k = 0..kMaxD+1
constexpr long long kBinomSat = 1LL << 62;
constexpr long long kMaxCells = 1LL << 24;  // largest contingency table (cells)
constexpr int kMaxVars = 32767;           // neighbour positions are stored in 16 bits
constexpr int kTestThreads = 256;         // threads of a test CTA
constexpr int kBigThreads = 1024;         // threads of a CTA of the big-table class
constexpr int kBaseSmem = 512;            // pass bases cached in shared memory

// device status bits
constexpr unsigned kStatusTooBig = 1u;    // table over kMaxCells or scratch too small
constexpr unsigned kStatusNumeric = 2u;   // p-value iteration hit its cap
constexpr unsigned kStatusSepPool = 4u;   // separating-set pool overflow
constexpr unsigned kStatusEdges = 8u;     // edge list overflow
constexpr unsigned kStatusTimeout = 16u;  // a bounded device wait gave up
constexpr unsigned kStatusScratch = 32u;  // a table needed more global scratch than allocated
constexpr int kMaxArityPairs = 256;       // arity bound of the depth-0 pair epilogue
// Depths 0 and 1 from one-hot bit planes: largest arity (kMargMaxArity - 1
// planes per variable; the x and y values of a test share one warp's lanes).
constexpr int kMargMaxArity = 5;
constexpr int kMargThreads = 256;          // threads of a k_pool_marg CTA

// One learning problem (one data set).  Arrays are device pointers.
struct ProblemDev {
    const uint8_t* data;   // [n][ld] uint8, variable-major, zero padded
    const uint8_t* ar;     // [n] arities
    uint8_t* adj;          // [n][n] current graph, 0/1
    int32_t* nbr;          // [n][n] snapshot a(v), ascending, deg[v] valid entries
    int32_t* deg;          // [n]
    int32_t* sep_len;      // [n][n] (entry i<j), -1 while adjacent
    int64_t* sep_off;      // [n][n] offset of the members in the shared pool
    int64_t ld;            // row stride (bytes), multiple of 256
    int32_t n;
    int32_t N;
    int32_t max_arity;
    int32_t nplanes;       // one-hot planes per variable: max_arity - 1, or 0 without planes
    // the pair tables of depth 0: table (i, j), i < j, at rows off[i].. and
    // columns off[j].. of gram; on the diagonal, the counts of single values
    const int32_t* off;    // [n] sum of the arities before each variable
    int32_t* gram;         // [gram_ld][gram_ld]
    int64_t gram_ld;
    // one-hot Gram over the values >= 1 (the cells of value 0 follow from it)
    const int32_t* roff;   // [n] first one-hot row of each variable: off[v] - v
    uint8_t* onehot;       // [rgram_ld][onehot_ld] E4M3 one-hot rows
    int32_t* rgram;        // [rgram_ld][rgram_ld] INT32 Gram (upper tile triangle)
    int64_t onehot_ld;     // padded samples (multiple of 128)
    int64_t rgram_ld;      // padded rows (multiple of 128)
    int32_t* eid;          // [n][n] edge of the current depth at each snapshot slot nbr[v][t]
    int32_t* npos;         // [n][n] npos[v][u] = index of u in nbr[v] (u adjacent to v in the snapshot)
    uint8_t* pk;           // [n][pk_ld] samples 4 bits each (depth-1 tensor-core path; arities <= 8)
    int64_t pk_ld;         // ld / 2
    // one-hot planes (every arity of the problem <= kMargMaxArity): bit s of
    // planes[(v * nplanes + a) * plane_ld + w] says that sample 32 w + s of
    // variable v has value a + 1.  plane_ld is a multiple of 4 words; bits past
    // the samples are zero; planes a >= r_v - 1 are not written.
    const uint32_t* planes;
    int64_t plane_ld;
};

// One edge i<j of the current depth with its rank space: ranks [0, cnt_i) are
// the X-side conditioning sets (subsets of a(i)\{j}), ranks [cnt_i, total) the
// Y-side ones (subsets of a(j)\{i}), each side in lexicographic order.
// posj = index of j in a(i), posi = index of i in a(j).
struct EdgeWork {
    int32_t prob, i, j;
    int16_t posj, posi;
    int64_t cnt_i, total;
};

// Per-depth codes of the autotuner (DepthCounters::tune).
constexpr int kTuneGroupMask = 0x3FF;
constexpr int kTuneNoBits = 0x400;

__host__ __device__ __forceinline__ int tune_code(const int* tune, int d)
{
    return tune && d >= 0 && d < 64 ? tune[d] : 0;
}

// Edge classes: tables that fit a warp's share of shared memory run on warp
// workers, the others on CTA workers.
constexpr int kClassWarp = 0;
constexpr int kClassCta = 1;
constexpr int kClassMarg = 2;   // not an edge class: the pool of depth 1 counted from one-hot planes

// Device-side state of the depth loop.  Per-depth fields are cleared by
// k_depth_begin; d, active, status and sep_used persist across depths.
// Per-depth record written by k_depth_end.
constexpr int kMaxDepthRecords = 64;
struct DepthRecord {
    long long edges, tests, tests_oracle, removed;
    long long test_samples;   // sum of N over the sequential order's tests (their problems' sample counts)
    long long popc_work;      // popcounts of the tests counted from one-hot planes (counted cells x 32-sample words)
    long long smem_updates;   // shared-memory histogram updates (samples of the tests counted by histogram)
    // device clock (ns): depth start (snapshot), test kernels start and end,
    // depth end; 0 where a kernel of the depth did not run
    unsigned long long t_begin, t_tests, t_tests_end, t_end;
};

struct DepthCounters {
    unsigned long long n_edges[2];      // edges per class
    unsigned long long maxc[2];         // largest chunk count per class
    unsigned long long next_item[2];    // work-pool claim counters
    unsigned long long total_items[2];  // work items per class
    unsigned long long tests;           // CI tests executed
    unsigned long long tests_oracle;    // tests of the sequential order (gs = 1)
    unsigned long long test_samples;    // sum over those tests of their problem's N
    unsigned long long popc_work;       // executed counting work: popcounts (one-hot planes)
    unsigned long long smem_updates;    // executed counting work: histogram updates (samples)
    unsigned long long removed;         // edges removed
    unsigned long long max_cells[2];    // upper bound of table cells per class
    unsigned long long sep_used;        // separating-set pool entries in use (persists)
    unsigned int status;                // error bits (persists)
    int d;                              // current depth (persists)
    int active;                         // 1 while Algorithm 1 continues (persists); -1: the persistent loop handed over
    int gsel;                           // group size of the small-table class this depth
    int need_cells;                     // largest table that missed the global scratch (persists)
    int gs;                             // ranks per chunk this depth (set by k_edges)
    unsigned long long adj_ends;        // sum of the snapshot degrees (twice the live edges)
    unsigned long long nbr_claim;       // vertex claims of the depth-1 tensor-core kernel
    unsigned long long max_total[2];    // largest rank count of an edge per class
    int split[2];                       // sample parts per test per class (1 = whole tests)
    int wide;                           // the big-table class runs on k_pool_big (0: k_pool_mid)
    int whole;                          // depth 1 from one-hot planes: an item is a whole edge (set by k_edges)
    unsigned int beat;                  // persistent loop: ranks begun after an item's first (its barriers wait on while
                                        // this or next_item moves)
    float cost[2];                      // estimated cycles of the depth's tests per class (choose_pool)
    int hand_over;                      // persistent loop: a table of this depth does not fit its shared memory
    int direct;                         // 1: item w is chunk w / E of the class's edge w mod E (empty past its last)
    DepthRecord* rec;                   // per-depth records (persists)
    const int* tune;                    // per-depth choices of the autotuner, or nullptr (persists):
                                        // kTuneGroupMask = threads per test of the small-table class (0: cost
                                        // model), kTuneNoBits = byte histograms only at that depth
};

// Tests split by samples: when a depth has few tests against the groups, every
// test is counted by `split` groups over disjoint sample ranges; each part adds
// its table into a zero global table of the test, and the part that finishes
// last decides and zeroes the table again.
constexpr int kMaxSplit = 16;
constexpr long long kSplitMinSamples = 4096;   // samples per part at least
constexpr long long kSplitItems = 4096;        // tests split at once at most

// Passes of the work pool are capped: an edge with more ranks than
// kMaxPasses * gs takes chunks of ceil(total / kMaxPasses) ranks.
constexpr long long kMaxPasses = 4096;

__host__ __device__ __forceinline__ long long chunk_ranks(long long total, int gs)
{
    const long long c = (total + kMaxPasses - 1) / kMaxPasses;
    return c > gs ? c : gs;
}

__host__ __device__ __forceinline__ long long chunk_count(long long total, int gs)
{
    const long long c = chunk_ranks(total, gs);
    return (total + c - 1) / c;
}

// Order key of an edge that is one work item of k_pool_marg, 1 .. kMaxPasses,
// descending: edges of one counting shape (the endpoints' arities) together, so
// that the warps of an SM run the same loop and its instructions stay cached;
// within a shape the longest (tests times samples, 8 steps per octave) first.
__device__ __forceinline__ long long edge_item_key(long long total, int N, int ra, int rb)
{
    const int A = ra > rb ? ra : rb, B = ra > rb ? rb : ra;        // 2 <= B <= A <= kMargMaxArity
    const int shape = (A - 2) * (A - 1) / 2 + (B - 2);             // 0 .. 9
    int w = (__float_as_int((float)total * (float)N) >> 20) - (127 << 3);
    w = w < 0 ? 0 : w > 399 ? 399 : w;
    return (long long)shape * 400 + w + 1;
}

// Per-class arguments of the ordering scan.
struct ScanClass {
    const unsigned long long* hist;   // chunk-count histogram of the class
    unsigned long long* alive;        // [maxc + 1] edges with more than k chunks
    unsigned long long* base;         // [maxc + 1] first item of pass k
    long long groups[4];              // groups of 32, 64, 128, 256 threads the class's pool runs
    long long smem_ints;              // shared ints of one pool CTA of the class
    long long mid_ints;               // big-table class: the same of a k_pool_mid CTA (0: no such kernel)
};

// Cache of critical values, see fbn_device.cuh.
struct CritTableDev {
    long long* keys;
    double* vals;
    int cap;
    int dense_n;           // df < dense_n: dense[df], 0 until a test computes it
    double* dense;
    float2* dense_f;       // df < dense_n: the float bracket (largest float <= crit, smallest >= crit), 0 until set
    long long* dense_q;    // df < dense_n: floor(crit / 2) in units of 2^-kLutBits, 0 until set
};

// Work pool of one depth and one edge class.  Sizes, the depth and the class
// sub-array come from the DepthCounters on the device.
struct PoolArgs {
    const ProblemDev* probs;
    const EdgeWork* edges;            // whole edge array (class 0 from the front, class 1 from the back)
    unsigned long long* min_accept;   // per edge, lowest accepting rank, init = total
    long long edge_cap;
    const int32_t* sorted;            // class edges by chunk count, descending
    const unsigned long long* base;   // [maxc + 1] first item of pass k
    DepthCounters* ctr;
    const long long* binom;           // [binom_rows][kBinomCols]
    int* gscratch;                    // global tables, gscratch_ints per group
    long long gscratch_ints;
    CritTableDev crit;
    int32_t cls;
    int32_t hand_over;                // 1: the persistent loop (a table over its shared memory ends the loop)
    int32_t smem_ints;
    int32_t binom_rows;
    double alpha;
    int* split_tab;                   // [kSplitItems][split_stride] zero global tables of split tests
    unsigned* split_ticket;           // [kSplitItems] parts finished per test, zero between uses
    long long split_stride;           // ints per split table
    int32_t stat;                     // CI statistic: 0 = G^2, 1 = Pearson X^2
    int32_t df_mode;                  // degrees of freedom: 0 = declared arities, 1 = observed table
    const long long* lut;             // n ln n in units of 2^-kLutBits up to the largest N, or nullptr: FP32 terms
    long long lut_err;                // bound of an entry's error, in its units
};

// Shared ints -> largest table a group's slice takes: the cells alone with the
// n ln n table, else the cells and their marginals (at most 1.25 C as r_x, r_y
// >= 2).
__host__ __device__ __forceinline__ long long slice_cells(long long slice_ints, bool need_marg)
{
    return need_marg ? (slice_ints - 8) * 4 / 9 : slice_ints;
}

}  // namespace fbn
