// fbn_api.cu -- host engine and C ABI (include/fbn.h) of the GB300 PC-stable
// skeleton library.  The depth loop of Algorithm 1 is set up here; the steps of a depth
// (snapshot, edge list, CI tests, removal) are kernels in fbn_kernels.cu, the
// Gram and pools' files, or for small calls phases of one kernel (fbn_loop.cu).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/fbn.h"
#include "fbn_ci.cuh"
#include "fbn_gram.h"
#include "fbn_loop.h"
#include "fbn_nbr.h"
#include "fbn_sepsets.h"
#include "fbn_launch.h"

using namespace fbn;

namespace {

thread_local std::string g_create_error;

constexpr size_t kSmemBytes = 100 * 1024;     // dynamic shared memory of a CTA test group: 2 CTAs / SM with the ~9 KB static
constexpr long long kSplitStride = 4096;        // cells of a split test's global table at most
constexpr size_t kWarpSmemBytes = 64 * 1024;  // dynamic shared memory of a CTA of the small-table pool (2 CTAs / SM)
constexpr size_t kBigSmemBytes = 200 * 1024;  // the same of the big-table pool (one CTA of 1,024 threads / SM)
// Variables of a call whose skeleton runs as one persistent kernel; above, the
// kernels of a depth as a graph: with more variables the phases fill the chip
// and a depth's fixed cost (37-41 us as kernels, 25-30 in the loop) no longer
// shows.  Learning and reading 20 variables x 5,000 samples 282 -> 182 us, 40 x
// 50,000 405 -> 310 us, 101 x 9,973 460 -> 385 us.  Up to kLoopOneCta variables
// one CTA per SM instead of two (20 variables: 157 us against 170 to learn; 101:
// 359 both, with depth 1 at 64 against 49 us).
constexpr int kLoopVertices = 512;
constexpr int kLoopOneCta = 32;

// Persistent calls of this process under way per device, those of other threads
// included.  All CTAs of such a call are resident at once, so a grid that fills the
// chip makes the calls of several threads wait for one another; each takes its share
// of the CTAs instead (the results do not depend on the grid), at least a quarter of
// the SMs: below, a call lasts as many times longer as there are fewer CTAs.  Calls
// per second of 1 / 2 / 4 / 8 threads, 101 variables x 9,973 samples: grids that fill
// the chip 3,215 3,403 3,402 3,394, one CTA on every second SM 2,460 4,839 8,556
// 8,842, on every fourth 1,910 3,784 7,386 12,858; the kernels of a depth as a graph
// 2,480 3,770 4,980 6,150.
constexpr int kLoopDevices = 64;
std::atomic<int> g_loops[kLoopDevices];

class LoopShare {
public:
    LoopShare(int device, bool take) : n_(take && device < kLoopDevices ? &g_loops[device] : nullptr)
    {
        if (n_) calls_ = n_->fetch_add(1) + 1;
    }
    ~LoopShare()
    {
        if (n_) n_->fetch_sub(1);
    }
    LoopShare(const LoopShare&) = delete;
    LoopShare& operator=(const LoopShare&) = delete;
    int grid(int full, int sms) const
    {
        int g = full;
        for (int c = 1; c < calls_ && g / 2 >= sms / 4; c *= 2) g /= 2;
        return g;
    }

private:
    std::atomic<int>* n_;
    int calls_ = 1;
};
constexpr size_t kAdjStageBytes = (size_t)16 << 20;   // pinned bytes a call's graphs pass through at most
constexpr int kCritCap = 8192;                // critical-value cache slots (power of two)
constexpr int kCritDense = 8192;              // critical values kept in a dense table: df < kCritDense

template <typename T>
cudaError_t dalloc(T** p, size_t count)
{
    *p = nullptr;
    if (count == 0) count = 1;
    return cudaMalloc((void**)p, count * sizeof(T));
}

void dfree(void* p)
{
    if (p) cudaFree(p);
}

// ---- small kernels of the host engine ------------------------------------
// One pass over new samples (a row per grid.y): into the padded store (data;
// nullptr: they are there already), the first value at or above its arity
// (row-major index over n x N), and the one-hot planes (nplanes > 0).  The
// samples come from any device-addressable memory, pinned host memory included,
// at any alignment: a CTA reads its 8,192 samples as whole aligned 16-byte words
// into shared memory and every thread shifts its 32 samples out of it.  Bounded
// by the host link (206 GB/s measured): one pass per data set, where a strided
// copy, a check and the planes took 40 us for 2.4 MB, three times its transfer.
constexpr int kIngestSamples = 8192;   // per CTA and step: 32 a thread

__global__ void __launch_bounds__(256) k_ingest(const uint8_t* src, int64_t stride, const uint8_t* src_end, int64_t N,
                                                int64_t ld, const uint8_t* __restrict__ ar, int nplanes, int64_t wp,
                                                uint8_t* data, uint32_t* __restrict__ planes,
                                                unsigned long long* first_bad)
{
    constexpr int kWords = kIngestSamples / 4 + 4;
    __shared__ unsigned s_w[kWords + kWords / 32 + 1];   // word i at i + i / 32: no bank conflicts at 8 words a thread
    const int v = blockIdx.y, tid = threadIdx.x;
    const int r = ar[v];
    const unsigned rr = 0x01010101u * (unsigned)r;
    const int values = nplanes > 0 ? r - 1 : 0;
    const long long words = data ? ld / 32 : wp;
    for (long long s0 = (long long)blockIdx.x * kIngestSamples; s0 < words * 32; s0 += (long long)gridDim.x * kIngestSamples) {
        const long long left = N - s0;
        const int cnt = left <= 0 ? 0 : left < kIngestSamples ? (int)left : kIngestSamples;
        const uint8_t* at = src + v * stride + s0;
        const int skip = (int)((uintptr_t)at & 15);
        const uint8_t* at0 = at - skip;
        for (int c = tid; c < (cnt ? (skip + cnt + 15) / 16 : 0); c += 256) {
            const uint8_t* p = at0 + 16 * c;
            unsigned q[4] = {0u, 0u, 0u, 0u};
            if (p >= src && p + 16 <= src_end) {
                const uint4 t = *reinterpret_cast<const uint4*>(p);
                q[0] = t.x; q[1] = t.y; q[2] = t.z; q[3] = t.w;
            } else {   // the buffer's first or last word
                for (int b = 0; b < 16; ++b)
                    if (p + b >= src && p + b < src_end) q[b >> 2] |= (unsigned)p[b] << ((b & 3) * 8);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) s_w[4 * c + k + (4 * c + k) / 32] = q[k];
        }
        __syncthreads();
        const long long w = s0 / 32 + tid;
        if (w < words) {
            const int i0 = (skip + 32 * tid) >> 2, sh = (skip & 3) * 8;
            const long long have = N - w * 32;
            unsigned x[9], q[8];
#pragma unroll
            for (int k = 0; k < 9; ++k) x[k] = s_w[i0 + k + (i0 + k) / 32];
            unsigned bad = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const long long m = have - 4 * k;   // samples of this word below N
                q[k] = __funnelshift_r(x[k], x[k + 1], sh) & (m >= 4 ? ~0u : m <= 0 ? 0u : (1u << (8 * (int)m)) - 1u);
                bad |= __vcmpgeu4(q[k], rr);
            }
            if (data) {
                uint4* d = reinterpret_cast<uint4*>(data + v * ld + w * 32);
                d[0] = make_uint4(q[0], q[1], q[2], q[3]);
                d[1] = make_uint4(q[4], q[5], q[6], q[7]);
            }
            if (bad) {
                for (int k = 0; k < 32; ++k)
                    if (((q[k >> 2] >> ((k & 3) * 8)) & 0xFFu) >= (unsigned)r) {
                        atomicMin(first_bad, (unsigned long long)v * (unsigned long long)N + (unsigned long long)(w * 32 + k));
                        break;
                    }
            }
            if (w < wp)
                for (int y = 1; y <= values; ++y) {
                    unsigned m = 0;
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        m |= (((__vcmpeq4(q[k], 0x01010101u * (unsigned)y) & 0x08040201u) * 0x01010101u) >> 24) << (4 * k);
                    planes[((long long)v * nplanes + y - 1) * wp + w] = m;
                }
        }
        __syncthreads();
    }
}

// Adjacencies of up to kAdjJob problems into pinned host memory, 16 bytes per
// thread and step.  A batch's graphs went to the caller's pageable memory one
// copy each, some 14 us apiece: 256 problems 17.4 ms to learn, through the pinned buffer 15.5;
// 20 problems 2.0 -> 1.84 ms.
constexpr int kAdjJob = 64;
struct AdjJob {
    const uint8_t* src[kAdjJob];   // n x n bytes, allocated in whole 16-byte words
    long long words[kAdjJob];      // 16-byte words
    long long off[kAdjJob];        // first word in dst
};

__global__ void __launch_bounds__(256) k_adj_out(AdjJob j, uint4* __restrict__ dst)
{
    const uint4* s = reinterpret_cast<const uint4*>(j.src[blockIdx.y]);
    uint4* d = dst + j.off[blockIdx.y];
    for (long long w = (long long)blockIdx.x * blockDim.x + threadIdx.x; w < j.words[blockIdx.y];
         w += (long long)gridDim.x * blockDim.x)
        d[w] = s[w];
}

// n ln n for n < count, in units of 2^-kLutBits (see grp_g2_lut).
__global__ void k_lut(long long* lut, int count)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n < count) lut[n] = n < 2 ? 0 : __double2ll_rn((double)n * log((double)n) * 68719476736.0);
}

__global__ void k_init_graph(const ProblemDev* probs, const int32_t* vtx_prob, const int32_t* vtx_first,
                             int total_vertices)
{
    const int g = blockIdx.x;
    if (g >= total_vertices) return;
    const int p = vtx_prob[g];
    const ProblemDev P = probs[p];
    const int i = g - vtx_first[p];
    for (int j = threadIdx.x; j < P.n; j += blockDim.x) {
        P.adj[(long long)i * P.n + j] = (uint8_t)(i != j);
        P.sep_len[(long long)i * P.n + j] = -1;
        P.sep_off[(long long)i * P.n + j] = 0;
    }
}

}  // namespace

// Pinned host memory that holds exported separating sets: the workspace's until
// it exports again, and every handle's whose sets lie in it.
struct HostStage {
    uint8_t* p = nullptr;
    uint8_t* dev = nullptr;   // as the device addresses it
    size_t cap = 0;
    ~HostStage()
    {
        if (p) cudaFreeHost(p);
    }
};

// ---- workspace shared by the depth loop ----------------------------------
struct Workspace {
    long long edge_cap = 0;
    EdgeWork* edges = nullptr;
    unsigned long long* min_accept = nullptr;
    int32_t* sorted = nullptr;
    long long ord_cap = 0;
    unsigned long long *hist = nullptr, *alive = nullptr, *base = nullptr, *cursor = nullptr;
    DepthCounters* d_ctr = nullptr;
    DepthCounters* h_ctr = nullptr;   // pinned
    long long* binom = nullptr;
    int brows = 0;
    int vtx_cap = 0, prob_cap = 0;
    int32_t *vtx_prob = nullptr, *vtx_first = nullptr;
    ProblemDev* probs = nullptr;
    int32_t* sep_pool = nullptr;
    long long sep_cap = 0;
    int* gscratch = nullptr;
    long long gscratch_total = 0;
    long long* crit_keys = nullptr;
    double* crit_vals = nullptr;
    double* crit_dense = nullptr;
    float2* crit_dense_f = nullptr;
    long long* crit_dense_q = nullptr;
    long long* lut = nullptr;                       // n ln n up to the largest N seen (kLutMaxN at most)
    long long lut_n = 0;
    double crit_alpha = -1.0;
    cudaEvent_t kev[2 * FBN_MAX_DEPTHS + 2] = {};   // the Gram's window at the end
    DepthRecord* d_rec = nullptr;
    DepthRecord* h_rec = nullptr;                   // pinned
    long long gs_cells = 0;                         // cells per group of the global scratch
    // one-hot Gram of a whole batch
    uint8_t* gram_E = nullptr;                      // one-hot matrices, problem after problem
    long long gram_E_cap = 0;
    int32_t* gram_G = nullptr;                      // pair tables, problem after problem
    long long gram_G_cap = 0;
    int32_t* gram_R = nullptr;                      // Grams over the values >= 1, problem after problem
    long long gram_R_cap = 0, gram_R_used = 0;
    uint8_t* gram_maps = nullptr;                   // tensor maps, one per problem
    long long gram_maps_cap = 0;
    int4* gram_units = nullptr;
    long long gram_units_cap = 0;
    // samples 4 bits each, problem after problem (depth 1 on the tensor cores)
    uint8_t* pk = nullptr;
    long long pk_cap = 0;
    // global tables of tests split by samples; zero between uses (cleared
    // again when a call did not run to its end)
    int* split_tab = nullptr;
    unsigned* split_ticket = nullptr;
    bool split_dirty = false;
    // per-depth choices of the autotuner on the device, as last uploaded
    int* d_tune = nullptr;
    std::vector<int> tune_loaded;
    // sharded skeletons: this process's edges, removal records, their count
    uint8_t* d_owned = nullptr;
    long long owned_cap = 0;
    long long* d_shard = nullptr;
    long long shard_cap = 0;
    unsigned long long* d_shard_count = nullptr;
    // launch geometry of the device, fixed once (kernel attributes set)
    int dev_sms = 0, grid_small = 0, grid_big = 0, grid_marg = 0, grid_loop = 0;
    // the problem descriptors and vertex maps as last uploaded (skipped when
    // unchanged), staged through pinned memory
    std::vector<uint8_t> up_last;
    uint8_t* h_up = nullptr;
    size_t h_up_cap = 0;
    // pinned staging of the separating-set export: totals, then the arrays
    long long* h_tot = nullptr;
    size_t h_tot_cap = 0;
    std::shared_ptr<HostStage> stage;
    unsigned long long *d_bads = nullptr, *h_bads = nullptr;   // first bad values of a batch of uploads
    size_t bad_cap = 0;
    unsigned* d_bar = nullptr;                      // barrier of the persistent loop
    unsigned* h_left = nullptr;                     // pinned: how the loop ended early (LoopArgs::left)
    unsigned* d_bits = nullptr;                     // its adjacency bit matrix
    uint8_t* h_adj = nullptr;                       // pinned: the adjacency it leaves
    size_t h_adj_cap = 0;
    int gram_n_units = 0, gram_unit_slices = 0;
    std::vector<uint8_t> h_maps;
    // one-hot layout of the last prepare_gram and the last one whose pad rows
    // were zeroed (k_onehot writes only the rows below M)
    std::vector<long long> gram_layout, gram_zeroed;
    // the graph of the generic depths (a device-driven while loop)
    cudaGraphExec_t loop = nullptr;
    std::vector<uint8_t> graph_key;
    cudaEvent_t tev[2] = {};   // window of the neighbourhood product
    bool events = false;

    void release()
    {
        dfree(edges); dfree(min_accept); dfree(sorted);
        dfree(hist); dfree(alive); dfree(base); dfree(cursor);
        dfree(d_ctr);
        if (h_ctr) cudaFreeHost(h_ctr);
        dfree(binom); dfree(vtx_prob); dfree(vtx_first); dfree(probs);
        dfree(sep_pool); dfree(gscratch); dfree(crit_keys); dfree(crit_vals); dfree(crit_dense);
        dfree(crit_dense_f); dfree(crit_dense_q); dfree(lut);
        dfree(gram_E); dfree(gram_G); dfree(gram_R); dfree(gram_maps); dfree(gram_units); dfree(pk);
        dfree(split_tab); dfree(split_ticket); dfree(d_tune);
        dfree(d_owned); dfree(d_shard); dfree(d_shard_count);
        if (events) {
            for (auto& e : kev) cudaEventDestroy(e);
            for (auto& e : tev) cudaEventDestroy(e);
        }
        if (loop) cudaGraphExecDestroy(loop);
        dfree(d_rec);
        if (h_rec) cudaFreeHost(h_rec);
        if (h_up) cudaFreeHost(h_up);
        if (h_tot) cudaFreeHost(h_tot);
        if (h_adj) cudaFreeHost(h_adj);
        if (h_bads) cudaFreeHost(h_bads);
        dfree(d_bads);
        dfree(d_bar); dfree(d_bits);
        if (h_left) cudaFreeHost(h_left);
        h_maps.clear();
        gram_E = nullptr; gram_G = nullptr; gram_R = nullptr; gram_maps = nullptr; gram_units = nullptr; pk = nullptr;
        split_tab = nullptr; split_ticket = nullptr;
        *this = Workspace();
    }
};

// A device array released when its last holder lets go.
struct DeviceInts {
    int32_t* d = nullptr;
    long long n = 0;
    cudaEvent_t ready = nullptr;        // after the copy that fills d, on the batch's stream
    std::vector<fbn_handle*> members;   // the handles whose sets live here (a batch)
    ~DeviceInts()
    {
        if (d) cudaFree(d);
        if (ready) cudaEventDestroy(ready);
    }
};

struct fbn_handle {
    int device = 0;
    cudaStream_t own_stream = nullptr;
    cudaStream_t stream = nullptr;
    fbn_options opt{};
    int n = 0;
    int64_t N = 0, ld = 0;
    int max_arity = 0;
    std::vector<uint8_t> h_ar;
    uint8_t* d_data = nullptr;
    uint32_t* d_planes = nullptr;       // one-hot planes (see k_ingest), none above arity kMargMaxArity
    int nplanes = 0;                    // planes per variable
    int64_t plane_ld = 0;               // words per plane, a multiple of 4
    uint8_t* d_ar = nullptr;
    uint8_t* d_adj = nullptr;
    int32_t* d_nbr = nullptr;
    int32_t* d_eid = nullptr;
    int32_t* d_npos = nullptr;
    int32_t* d_deg = nullptr;
    int32_t* d_sep_len = nullptr;
    int64_t* d_sep_off = nullptr;
    // explicit tests: the kernel writes its results and small tables straight
    // into pinned host memory; larger tables and global tables on the device
    double* h_ci_out = nullptr;   // pinned: statistic, df, p
    unsigned* h_status = nullptr; // pinned
    double* ci_out_dev = nullptr; // the two as the device addresses them
    unsigned* status_dev = nullptr;
    int ci_cluster_max = 0;       // 0: the kernel's limits are not set yet
    int32_t* h_table = nullptr;   // pinned
    long long h_table_cap = 0;
    int32_t* d_table = nullptr;
    long long table_cap = 0;
    int* d_gscratch = nullptr;
    long long gscratch_ints = 0;
    unsigned long long* d_bad = nullptr;   // first out-of-range value of an upload
    unsigned* d_status = nullptr;
    // one-hot Gram (depth 0 on tensor cores)
    int M = 0;                          // sum of arities
    int Mp = 0;                         // M padded to the tile
    int Mr = 0;                         // M - n (values >= 1) padded to the tile
    long long K = 0;                    // samples padded to the stage width
    int32_t* d_off = nullptr;           // [n] sum of the arities before each variable; [n] the same of arities - 1
    // results of the last skeleton
    bool learnt = false;
    bool sep_pending = false;           // separating sets still only on the device
    unsigned long long sep_pool_used = 0;
    // members of a batch's separating sets: a device copy of the batch's
    // shared pool, held by every handle of that batch until it learns again
    std::shared_ptr<DeviceInts> sep_snap;
    // separating sets on the host, CSR in pinned memory: removed pairs (i < j)
    // ascending, their member offsets, the members
    std::shared_ptr<HostStage> csr_hold;
    const int32_t* csr_pairs = nullptr;
    const int64_t* csr_offs = nullptr;
    const int32_t* csr_members = nullptr;
    long long csr_R = 0, csr_M = 0;
    // row counts of the compaction on the device, [2n]
    long long* d_sep_cnt = nullptr;
    fbn_stats stats{};
    // the autotuner's choices (empty: the fixed rules): a per-depth code
    // (kTuneGroupMask, kTuneNoBits) and how depth 0 counts (0: the rule)
    std::vector<int> tune;
    int tune_depth0 = 0;
    Workspace ws;
    std::string err;
};

namespace {

int fail(fbn_handle* h, int code, const char* fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    if (h) h->err = buf; else g_create_error = buf;
    return code;
}

#define CK(call)                                                                       \
    do {                                                                               \
        cudaError_t e_ = (call);                                                       \
        if (e_ != cudaSuccess)                                                         \
            return fail(h, e_ == cudaErrorMemoryAllocation ? FBN_ENOMEM : FBN_ECUDA,   \
                        "%s: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__); \
    } while (0)


int ensure_order(fbn_handle* h, Workspace& ws, long long maxc);

int grow_workspace(fbn_handle* h, Workspace& ws, long long edge_cap, int max_n, int nprob, int total_vtx)
{
    if (!ws.d_ctr) {
        CK(dalloc(&ws.d_ctr, 1));
        CK(cudaMallocHost((void**)&ws.h_ctr, sizeof(DepthCounters)));
        for (auto& e : ws.kev) CK(cudaEventCreate(&e));
        for (auto& e : ws.tev) CK(cudaEventCreate(&e));
        ws.events = true;
        CK(dalloc(&ws.d_rec, kMaxDepthRecords));
        CK(cudaMallocHost((void**)&ws.h_rec, kMaxDepthRecords * sizeof(DepthRecord)));
        const int orc = ensure_order(h, ws, kMaxPasses);
        if (orc) return orc;
        CK(dalloc(&ws.crit_keys, kCritCap));
        CK(dalloc(&ws.crit_vals, kCritCap));
        CK(dalloc(&ws.crit_dense, kCritDense));
        CK(dalloc(&ws.crit_dense_f, kCritDense));
        CK(dalloc(&ws.crit_dense_q, kCritDense));
        CK(dalloc(&ws.split_tab, kSplitItems * kSplitStride));
        CK(dalloc(&ws.split_ticket, kSplitItems));
        ws.split_dirty = true;
        CK(dalloc(&ws.d_tune, kMaxDepthRecords));
    }
    if (edge_cap > ws.edge_cap) {
        dfree(ws.edges); dfree(ws.min_accept); dfree(ws.sorted);
        ws.edges = nullptr; ws.min_accept = nullptr; ws.sorted = nullptr; ws.edge_cap = 0;
        CK(dalloc(&ws.edges, edge_cap));
        CK(dalloc(&ws.min_accept, edge_cap));
        CK(dalloc(&ws.sorted, edge_cap));
        ws.edge_cap = edge_cap;
    }
    if (max_n + 1 > ws.brows) {
        dfree(ws.binom);
        ws.binom = nullptr;
        const int rows = max_n + 1;
        std::vector<long long> B((size_t)rows * kBinomCols, 0);
        for (int nn = 0; nn < rows; ++nn) {
            B[(size_t)nn * kBinomCols] = 1;
            for (int k = 1; k < kBinomCols; ++k) {
                if (nn == 0) break;
                const long long a = B[(size_t)(nn - 1) * kBinomCols + k - 1];
                const long long b = B[(size_t)(nn - 1) * kBinomCols + k];
                long long s = a + b;
                if (s > kBinomSat || s < 0) s = kBinomSat;
                B[(size_t)nn * kBinomCols + k] = s;
            }
        }
        CK(dalloc(&ws.binom, B.size()));
        // on the handle's stream: it does not wait for the legacy one (as below)
        CK(cudaMemcpyAsync(ws.binom, B.data(), B.size() * sizeof(long long), cudaMemcpyHostToDevice, h->stream));
        CK(cudaStreamSynchronize(h->stream));
        ws.brows = rows;
    }
    if (total_vtx > ws.vtx_cap) {
        dfree(ws.vtx_prob); dfree(ws.vtx_first);
        ws.vtx_prob = nullptr; ws.vtx_first = nullptr; ws.vtx_cap = 0;
        CK(dalloc(&ws.vtx_prob, total_vtx));
        CK(dalloc(&ws.vtx_first, std::max(nprob, total_vtx)));
        ws.vtx_cap = total_vtx;
    }
    if (nprob > ws.prob_cap) {
        dfree(ws.probs);
        ws.probs = nullptr; ws.prob_cap = 0;
        CK(dalloc(&ws.probs, nprob));
        ws.prob_cap = nprob;
    }
    return FBN_OK;
}

int ensure_order(fbn_handle* h, Workspace& ws, long long maxc)
{
    if (maxc + 1 <= ws.ord_cap) return FBN_OK;
    dfree(ws.hist); dfree(ws.alive); dfree(ws.base); dfree(ws.cursor);
    ws.hist = ws.alive = ws.base = ws.cursor = nullptr;
    ws.ord_cap = 0;
    const long long cap = maxc + 1;   // per class; both classes side by side
    CK(dalloc(&ws.hist, 2 * cap));
    CK(dalloc(&ws.alive, 2 * cap));
    CK(dalloc(&ws.base, 2 * cap));
    CK(dalloc(&ws.cursor, 2 * cap));
    ws.ord_cap = cap;
    return FBN_OK;
}

int ensure_sep_pool(fbn_handle* h, Workspace& ws, long long need, long long used, cudaStream_t st)
{
    if (need <= ws.sep_cap) return FBN_OK;
    const long long cap = std::max(need, 2 * ws.sep_cap);
    int32_t* p = nullptr;
    CK(dalloc(&p, cap));
    if (ws.sep_pool && used > 0)
        CK(cudaMemcpyAsync(p, ws.sep_pool, used * sizeof(int32_t), cudaMemcpyDeviceToDevice, st));
    CK(cudaStreamSynchronize(st));
    dfree(ws.sep_pool);
    ws.sep_pool = p;
    ws.sep_cap = cap;
    return FBN_OK;
}

int ensure_gscratch(fbn_handle* h, Workspace& ws, long long total_ints)
{
    if (total_ints <= ws.gscratch_total) return FBN_OK;
    dfree(ws.gscratch);
    ws.gscratch = nullptr;
    ws.gscratch_total = 0;
    CK(dalloc(&ws.gscratch, total_ints));
    ws.gscratch_total = total_ints;
    return FBN_OK;
}

int check_status(fbn_handle* h, unsigned status)
{
    if (status & kStatusTooBig) return fail(h, FBN_ETOOBIG, "a contingency table exceeds %lld cells", kMaxCells);
    if (status & kStatusNumeric) return fail(h, FBN_ENUMERIC, "p-value iteration did not converge");
    if (status & kStatusSepPool) return fail(h, FBN_ECUDA, "separating-set pool overflow");
    if (status & kStatusEdges) return fail(h, FBN_ECUDA, "edge list overflow");
    if (status & kStatusTimeout) return fail(h, FBN_ETIMEOUT, "a bounded device wait gave up");
    if (status & kStatusScratch) return fail(h, FBN_ENOMEM, "global table scratch too small");
    return FBN_OK;
}

// The address at which kernels of `device` reach [p, p + bytes) in place: memory of
// the device or, with host, pinned host memory, from the first byte to the last;
// else nullptr (then a copy, which checks the range itself).
const void* device_range(const void* p, size_t bytes, int device, bool host)
{
    cudaPointerAttributes a{}, b{};
    const char* last = (const char*)p + (bytes ? bytes - 1 : 0);
    const bool ok = cudaPointerGetAttributes(&a, p) == cudaSuccess && a.devicePointer &&
                    ((host && a.type == cudaMemoryTypeHost) || (a.type == cudaMemoryTypeDevice && a.device == device)) &&
                    cudaPointerGetAttributes(&b, last) == cudaSuccess && b.type == a.type &&
                    (const char*)b.devicePointer - (const char*)a.devicePointer == last - (const char*)p;
    cudaGetLastError();
    return ok ? a.devicePointer : nullptr;
}

// New samples into the handle's store, with their check and planes; *bad (device,
// all ones before) receives the first bad value.  Pinned host memory and memory
// of the handle's device are read by the kernel itself; pageable memory (and
// any other) is copied first.
int ingest(fbn_handle* h, const uint8_t* data, unsigned long long* bad, cudaStream_t st)
{
    const uint8_t* src = (const uint8_t*)device_range(data, (size_t)h->n * h->N, h->device, true);
    int64_t stride = h->N;
    uint8_t* store = h->d_data;
    if (!src) {
        CK(cudaMemcpy2DAsync(h->d_data, h->ld, data, h->N, h->N, h->n, cudaMemcpyDefault, st));
        src = h->d_data;
        stride = h->ld;
        store = nullptr;
    }
    // grid.y is limited to 65,535: kMaxVars rows fit
    dim3 grid((unsigned)std::min<long long>((h->ld + kIngestSamples - 1) / kIngestSamples, 1024), h->n);
    k_ingest<<<grid, 256, 0, st>>>(src, stride, src + (h->n - 1) * stride + h->N, h->N, h->ld, h->d_ar, h->nplanes,
                                   h->plane_ld, store, h->d_planes, bad);
    CK(cudaGetLastError());
    return FBN_OK;
}

// Whether depth 0 runs as the one-hot Gram on tensor cores.
bool use_gram(fbn_handle* const* hs, int k, bool rule_only = false)
{
    const fbn_handle* h = hs[0];
    if (h->opt.depth0 == FBN_DEPTH0_GRAM) return true;
    if (h->opt.depth0 == FBN_DEPTH0_HIST) return false;
    if (!rule_only && h->tune_depth0) return h->tune_depth0 == FBN_DEPTH0_GRAM;
    long long M = 0, Nmax = 0;
    for (int p = 0; p < k; ++p) {
        M += hs[p]->M;
        Nmax = std::max<long long>(Nmax, hs[p]->N);
    }
    return M >= 512 && Nmax >= 4096;
}

// Depth 1 on the tensor cores: pool form, asked for, every arity within the
// kernel's bound.  The work pool stays the default: on the measured workloads
// it is faster, its early exit running about a quarter of the tests the
// neighbourhood product evaluates.
bool use_nbr1(fbn_handle* const* hs, int k)
{
    const fbn_handle* h = hs[0];
    if (h->opt.form == FBN_FORM_PLAIN || h->opt.depth1 != FBN_DEPTH1_TENSOR) return false;
    if (h->opt.statistic != FBN_STAT_G2 || h->opt.df_mode != FBN_DF_FIXED) return false;
    for (int p = 0; p < k; ++p)
        if (hs[p]->max_arity > nbr1_max_arity()) return false;
    return true;
}

// How the first depths of a skeleton call run.
struct DepthPlan {
    bool gram = false;    // depth 0 as the tensor-core Gram
    bool popc0 = false;   // depth 0 from one-hot planes (k_pairs_popc)
    bool marg1 = false;   // depth 1 from one-hot planes and depth 0's pair tables (k_pool_marg)
    bool nbr1 = false;    // depth 1 as the neighbourhood product
};

// The planes take every problem of the call or none (one pool per depth), at
// arities the planes hold; the caller may ask for histograms (count), and the
// autotuner for histograms at a depth.  A sharded skeleton counts every pair
// itself, without the Gram.
DepthPlan depth_plan(fbn_handle* const* hs, int k, bool shard)
{
    const fbn_handle* h = hs[0];
    DepthPlan p;
    if (h->opt.form == FBN_FORM_PLAIN) return p;
    p.gram = !shard && use_gram(hs, k);
    p.nbr1 = !shard && use_nbr1(hs, k);
    bool planes = h->opt.count != FBN_COUNT_HIST;
    for (int q = 0; q < k; ++q) planes = planes && hs[q]->nplanes > 0;
    auto hist_at = [&](int d) { return (size_t)d < h->tune.size() && (h->tune[d] & kTuneNoBits) != 0; };
    p.popc0 = planes && !p.gram && !hist_at(0);
    p.marg1 = planes && !p.nbr1 && (p.gram || p.popc0) && !hist_at(1);
    return p;
}

// Room for every problem's samples at 4 bits each; sets the problems' pk rows.
int prepare_pack(fbn_handle* const* hs, int k, Workspace& ws, ProblemDev* P)
{
    fbn_handle* h = hs[0];
    long long total = 0;
    for (int p = 0; p < k; ++p) total += (long long)hs[p]->n * (hs[p]->ld / 2);
    if (total > ws.pk_cap) {
        dfree(ws.pk);
        ws.pk = nullptr;
        ws.pk_cap = 0;
        CK(dalloc(&ws.pk, total));
        ws.pk_cap = total;
    }
    long long off = 0;
    for (int p = 0; p < k; ++p) {
        P[p].pk = ws.pk + off;
        P[p].pk_ld = hs[p]->ld / 2;
        off += (long long)hs[p]->n * (hs[p]->ld / 2);
    }
    return FBN_OK;
}

// Room for every problem's pair tables (the Gram layout); sets the problems'
// pointers.
int prepare_pairs(fbn_handle* const* hs, int k, Workspace& ws, ProblemDev* P)
{
    fbn_handle* h = hs[0];
    long long total = 0;
    for (int p = 0; p < k; ++p) total += (long long)hs[p]->Mp * hs[p]->Mp;
    if (total > ws.gram_G_cap) {
        dfree(ws.gram_G);
        ws.gram_G = nullptr;
        ws.gram_G_cap = 0;
        CK(dalloc(&ws.gram_G, total));
        ws.gram_G_cap = total;
    }
    long long go = 0;
    for (int p = 0; p < k; ++p) {
        P[p].off = hs[p]->d_off;
        P[p].gram = ws.gram_G + go;
        P[p].gram_ld = hs[p]->Mp;
        go += (long long)hs[p]->Mp * hs[p]->Mp;
    }
    return FBN_OK;
}

// Lay out the one-hot matrices and Grams of every problem in the workspace,
// set the problems' pointers, and upload one tensor map per problem and the
// work units (problem, tile pair, chunk), problem-major.
int prepare_gram(fbn_handle* const* hs, int k, Workspace& ws, ProblemDev* P)
{
    fbn_handle* h = hs[0];
    cudaStream_t st = h->stream;
    long long e_total = 0, r_total = 0;
    std::vector<long long> tiles(k), stages(k);
    for (int p = 0; p < k; ++p) {
        e_total += (long long)hs[p]->Mr * hs[p]->K;
        r_total += (long long)hs[p]->Mr * hs[p]->Mr;
        const int T = hs[p]->Mr / 128, T2 = (T + 1) / 2;
        for (int a = 0; a < T; ++a) tiles[p] += T2 - a / 2;
        stages[p] = hs[p]->K / 128;
    }
    if (r_total > ws.gram_R_cap) {
        dfree(ws.gram_R);
        ws.gram_R = nullptr;
        ws.gram_R_cap = 0;
        CK(dalloc(&ws.gram_R, r_total));
        ws.gram_R_cap = r_total;
    }
    ws.gram_R_used = r_total;
    int sms = 0;
    CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device));
    ws.gram_unit_slices = gram_unit_slices(tiles.data(), stages.data(), k, sms);
    if (e_total > ws.gram_E_cap) {
        dfree(ws.gram_E);
        ws.gram_E = nullptr;
        ws.gram_E_cap = 0;
        CK(dalloc(&ws.gram_E, e_total));
        ws.gram_E_cap = e_total;
    }
    const size_t mb = tensor_map_bytes();
    if ((long long)(k * mb) > ws.gram_maps_cap) {
        dfree(ws.gram_maps);
        ws.gram_maps = nullptr;
        ws.gram_maps_cap = 0;
        CK(dalloc(&ws.gram_maps, k * mb));
        ws.gram_maps_cap = (long long)(k * mb);
    }
    ws.h_maps.assign(k * mb, 0);
    std::vector<int4> units;
    long long eo = 0, ro = 0;
    ws.gram_layout.assign(1, (long long)(uintptr_t)ws.gram_E);
    for (int p = 0; p < k; ++p) {
        const fbn_handle* q = hs[p];
        P[p].onehot = ws.gram_E + eo;
        P[p].onehot_ld = q->K;
        P[p].off = q->d_off;
        P[p].roff = q->d_off + q->n;
        P[p].rgram = ws.gram_R + ro;
        P[p].rgram_ld = q->Mr;
        CK(encode_onehot_map(ws.h_maps.data() + p * mb, P[p].onehot, q->Mr, q->K));
        // 128-row tiles a against 256-row tiles b that reach the upper triangle
        const int T = q->Mr / 128, T2 = (T + 1) / 2, C = gram_chunks(q->K, ws.gram_unit_slices);
        for (int c = 0; c < C; ++c)
            for (int a = 0; a < T; ++a)
                for (int b = a / 2; b < T2; ++b) units.push_back(make_int4(p, a, b, c));
        ws.gram_layout.push_back(eo);
        ws.gram_layout.push_back(q->M);
        ws.gram_layout.push_back(q->Mr);
        ws.gram_layout.push_back(q->K);
        eo += (long long)q->Mr * q->K;
        ro += (long long)q->Mr * q->Mr;
    }
    if ((long long)units.size() > ws.gram_units_cap) {
        dfree(ws.gram_units);
        ws.gram_units = nullptr;
        ws.gram_units_cap = 0;
        CK(dalloc(&ws.gram_units, units.size()));
        ws.gram_units_cap = (long long)units.size();
    }
    ws.gram_n_units = (int)units.size();
    CK(cudaMemcpyAsync(ws.gram_maps, ws.h_maps.data(), k * mb, cudaMemcpyHostToDevice, st));
    CK(cudaMemcpyAsync(ws.gram_units, units.data(), units.size() * sizeof(int4), cudaMemcpyHostToDevice, st));
    return FBN_OK;
}

// One-hot matrices and their INT32 Grams (upper tile triangle) for the
// problems already in ws.probs (prepared by prepare_gram).
int run_gram(fbn_handle* h, Workspace& ws, int k, int total_vtx, unsigned* d_status, const DepthCounters* ctr = nullptr,
             cudaEvent_t ev0 = nullptr, cudaEvent_t ev1 = nullptr)
{
    cudaStream_t st = h->stream;
    int sms = 0;
    CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device));
    if (ws.gram_layout != ws.gram_zeroed) {   // pad rows stay zero while the layout holds
        CK(launch_zero_pad(ws.probs, k, st));
        ws.gram_zeroed = ws.gram_layout;
    }
    CK(launch_onehot(ws.probs, ws.vtx_prob, ws.vtx_first, total_vtx, ctr, st));
    CK(cudaMemsetAsync(ws.gram_R, 0, ws.gram_R_used * sizeof(int32_t), st));
    if (ev0) CK(cudaEventRecord(ev0, st));
    CK(launch_gram(ws.gram_maps, ws.gram_units, ws.gram_n_units, ws.gram_unit_slices, ws.probs, sms, d_status, h->opt.wait_limit, st));
    if (ev1) CK(cudaEventRecord(ev1, st));
    return FBN_OK;
}

// Move a handle to another separating-set snapshot (or to none).
void set_snapshot(fbn_handle* h, std::shared_ptr<DeviceInts> snap)
{
    if (h->sep_snap) {
        auto& m = h->sep_snap->members;
        m.erase(std::remove(m.begin(), m.end(), h), m.end());
    }
    h->sep_snap = std::move(snap);
    if (h->sep_snap) h->sep_snap->members.push_back(h);
}

// Grow a pinned host buffer (contents not kept).
template <class T>
cudaError_t grow_pinned(T** p, size_t* cap, size_t n)
{
    if (n <= *cap) return cudaSuccess;
    if (*p) cudaFreeHost(*p);
    *p = nullptr;
    *cap = 0;
    const cudaError_t e = cudaMallocHost((void**)p, std::max<size_t>(n, 1) * sizeof(T));
    if (e == cudaSuccess) *cap = n;
    return e;
}

// Pinned memory of at least `bytes` for an export; a new block when a handle
// still reads from the old one.
cudaError_t acquire_stage(Workspace& ws, size_t bytes)
{
    if (ws.stage && ws.stage.use_count() == 1 && ws.stage->cap >= bytes) return cudaSuccess;
    auto fresh = std::make_shared<HostStage>();
    cudaError_t e = cudaMallocHost((void**)&fresh->p, std::max<size_t>(bytes, 16));
    if (e == cudaSuccess) e = cudaHostGetDevicePointer((void**)&fresh->dev, fresh->p, 0);
    if (e != cudaSuccess) return e;
    fresh->cap = bytes;
    ws.stage = std::move(fresh);
    return cudaSuccess;
}

// A skeleton's CSR laid out for L pairs from an offset of the stage: pairs int32
// [2L], offsets int64 [L], members int32.
struct CsrPlace {
    size_t pairs, offs, members;
    CsrPlace(size_t at, long long L)
        : pairs(at), offs(at + 2 * (size_t)L * sizeof(int32_t)),
          members(at + (size_t)L * (2 * sizeof(int32_t) + sizeof(int64_t)))
    {
    }
    static size_t bytes(long long L, long long M)   // rounded to 16
    {
        return ((size_t)L * (2 * sizeof(int32_t) + sizeof(int64_t)) + (size_t)M * sizeof(int32_t) + 15) & ~(size_t)15;
    }
};

// The handle's sets are R pairs and M members at a place of the stage.
void take_csr(fbn_handle* q, const std::shared_ptr<HostStage>& stage, const CsrPlace& at, long long R, long long M)
{
    q->csr_hold = stage;
    q->csr_pairs = reinterpret_cast<const int32_t*>(stage->p + at.pairs);
    q->csr_offs = reinterpret_cast<const int64_t*>(stage->p + at.offs);
    q->csr_members = reinterpret_cast<const int32_t*>(stage->p + at.members);
    q->csr_R = R;
    q->csr_M = M;
    q->sep_pending = false;
}

// Results of the last skeleton are dropped.
void drop_sepsets(fbn_handle* q)
{
    q->sep_pending = false;
    q->csr_hold.reset();
    q->csr_pairs = q->csr_members = nullptr;
    q->csr_offs = nullptr;
    q->csr_R = q->csr_M = 0;
}

// The handle's separating sets as host CSR, compacted on the device by a
// kernel that writes the compact arrays straight into pinned host memory, where
// they stay.  One handle: sized by bounds known on the host (every pair removed;
// every pool entry its own), one synchronisation.  A handle of a batch: every
// member whose sets are still on the device, in two passes (row counts and
// totals; then the arrays), one synchronisation each.
int materialize_sepsets(fbn_handle* h, Workspace& ws)
{
    if (!h->sep_pending) return FBN_OK;
    CK(cudaSetDevice(h->device));
    cudaStream_t st = h->stream;
    std::vector<fbn_handle*> todo;
    if (h->sep_snap) {
        CK(cudaStreamWaitEvent(st, h->sep_snap->ready, 0));   // a member's stream need not be the batch's
        for (fbn_handle* q : h->sep_snap->members)
            if (q->sep_pending && q->device == h->device) todo.push_back(q);
    } else {
        todo.push_back(h);
    }
    const size_t k = todo.size();
    CK(grow_pinned(&ws.h_tot, &ws.h_tot_cap, 2 * k));
    long long* tot = nullptr;
    CK(cudaHostGetDevicePointer((void**)&tot, ws.h_tot, 0));
    std::vector<SepJob> jobs(k);
    for (size_t i = 0; i < k; ++i) {
        fbn_handle* q = todo[i];
        if (!q->d_sep_cnt) CK(dalloc(&q->d_sep_cnt, 2 * (size_t)q->n));
        SepJob& j = jobs[i];
        j = SepJob{};
        j.sep_len = q->d_sep_len;
        j.sep_off = q->d_sep_off;
        j.pool = q->sep_snap ? q->sep_snap->d : q->ws.sep_pool;
        j.n = q->n;
        j.cnt = q->d_sep_cnt;
        j.tot = tot + 2 * i;
    }
    auto place = [&](size_t i, const CsrPlace& at) {
        jobs[i].pairs = reinterpret_cast<int32_t*>(ws.stage->dev + at.pairs);
        jobs[i].offs = reinterpret_cast<int64_t*>(ws.stage->dev + at.offs);
        jobs[i].members = reinterpret_cast<int32_t*>(ws.stage->dev + at.members);
    };
    CK(launch_sep_count(jobs.data(), (int)k, st));
    if (k == 1) {
        fbn_handle* q = todo[0];
        const long long Rmax = (long long)q->n * (q->n - 1) / 2, Mmax = (long long)q->sep_pool_used;
        CK(acquire_stage(ws, CsrPlace::bytes(Rmax, Mmax)));
        const CsrPlace at(0, Rmax);
        place(0, at);
        CK(launch_sep_write(jobs.data(), 1, st));
        CK(cudaStreamSynchronize(st));
        if (ws.h_tot[0] > Rmax || ws.h_tot[1] > Mmax) return fail(h, FBN_ECUDA, "separating-set export over its bounds");
        take_csr(q, ws.stage, at, ws.h_tot[0], ws.h_tot[1]);
        return FBN_OK;
    }
    CK(cudaStreamSynchronize(st));
    std::vector<size_t> begin(k + 1, 0);
    for (size_t i = 0; i < k; ++i) begin[i + 1] = begin[i] + CsrPlace::bytes(ws.h_tot[2 * i], ws.h_tot[2 * i + 1]);
    CK(acquire_stage(ws, begin[k]));
    for (size_t i = 0; i < k; ++i) place(i, CsrPlace(begin[i], ws.h_tot[2 * i]));
    CK(launch_sep_write(jobs.data(), (int)k, st));
    CK(cudaStreamSynchronize(st));
    for (size_t i = 0; i < k; ++i)
        take_csr(todo[i], ws.stage, CsrPlace(begin[i], ws.h_tot[2 * i]), ws.h_tot[2 * i], ws.h_tot[2 * i + 1]);
    return FBN_OK;
}

// End of pair k's members.
int64_t csr_end(const fbn_handle* h, long long k) { return k + 1 < h->csr_R ? h->csr_offs[k + 1] : h->csr_M; }

// Index of the removed pair (i < j) in the handle's CSR, or -1.
long long find_sepset(const fbn_handle* h, int i, int j)
{
    long long lo = 0, hi = h->csr_R;   // pairs [0, R)
    while (lo < hi) {
        const long long mid = (lo + hi) >> 1;
        const int a = h->csr_pairs[2 * mid], b = h->csr_pairs[2 * mid + 1];
        if (a < i || (a == i && b < j)) lo = mid + 1; else hi = mid;
    }
    if (lo < h->csr_R && h->csr_pairs[2 * lo] == i && h->csr_pairs[2 * lo + 1] == j) return lo;
    return -1;
}

// Callbacks of a sharded skeleton (fbn_learn_skeleton_sharded).
struct ShardHooks {
    fbn_shard_own_fn own;
    fbn_shard_exchange_fn exchange;
    void* ctx;
};

// The depth loop of Algorithm 1 over one or more problems sharing a stream,
// one attempt.  Every kernel of a depth takes the depth and the sizes from the
// device counters.  *retry is set when a separating-set pool or global-table
// scratch turned out too small (both are grown before returning), or when a
// wait of the persistent loop ran out (*allow_loop is cleared: the depths then
// run as a graph, whose kernels wait for nothing).
int run_skeleton_once(fbn_handle* const* hs, int k, double alpha, int32_t max_depth, bool* retry, bool* allow_loop,
                      uint8_t* const* adj_out, const ShardHooks* shard = nullptr)
{
    fbn_handle* h = hs[0];
    Workspace& ws = h->ws;
    cudaStream_t st = h->stream;
    *retry = false;
    CK(cudaSetDevice(h->device));
    if (h->sep_snap) CK(cudaStreamWaitEvent(st, h->sep_snap->ready, 0));   // a batch's copy out of this pool, on another stream perhaps
    long long edge_cap = 0;
    int max_n = 0, total_vtx = 0;
    std::vector<ProblemDev> P(k);
    std::vector<int32_t> vtx_prob, vtx_first(k);
    for (int p = 0; p < k; ++p) {
        const fbn_handle* q = hs[p];
        edge_cap += (long long)q->n * (q->n - 1) / 2;
        max_n = std::max(max_n, q->n);
        vtx_first[p] = total_vtx;
        total_vtx += q->n;
        for (int v = 0; v < q->n; ++v) vtx_prob.push_back(p);
        ProblemDev& d = P[p];
        d.data = q->d_data; d.ar = q->d_ar; d.adj = q->d_adj; d.nbr = q->d_nbr; d.eid = q->d_eid; d.npos = q->d_npos; d.deg = q->d_deg;
        d.sep_len = q->d_sep_len; d.sep_off = q->d_sep_off; d.ld = q->ld; d.n = q->n; d.N = (int32_t)q->N;
        d.max_arity = q->max_arity; d.nplanes = q->nplanes;
        d.planes = q->d_planes; d.plane_ld = q->plane_ld;
    }
    int rc = grow_workspace(h, ws, edge_cap, max_n, k, total_vtx);
    if (rc) return rc;
    const bool plain = h->opt.form == FBN_FORM_PLAIN;
    if (shard && k != 1) return fail(h, FBN_EINVAL, "a sharded skeleton learns one problem");
    const DepthPlan plan = depth_plan(hs, k, shard != nullptr);
    const bool gram = plan.gram, nbr1 = plan.nbr1, popc0 = plan.popc0;
    const bool marg1 = plan.marg1 && max_depth != 0;
    if (shard) {   // this process's edges (n x n) and the depth's removal records (3 per edge at most)
        const long long nn = (long long)h->n * h->n;
        if (nn > ws.owned_cap) {
            dfree(ws.d_owned);
            ws.d_owned = nullptr;
            ws.owned_cap = 0;
            CK(dalloc(&ws.d_owned, nn));
            ws.owned_cap = nn;
        }
        if (edge_cap > ws.shard_cap) {
            dfree(ws.d_shard);
            ws.d_shard = nullptr;
            ws.shard_cap = 0;
            CK(dalloc(&ws.d_shard, 3 * edge_cap));
            ws.shard_cap = edge_cap;
        }
        if (!ws.d_shard_count) CK(dalloc(&ws.d_shard_count, 1));
    }
    if (nbr1) {
        rc = prepare_pack(hs, k, ws, P.data());
        if (rc) return rc;
    }
    if (gram) {
        rc = prepare_gram(hs, k, ws, P.data());
        if (rc) return rc;
    }
    if (popc0 || (gram && marg1)) {
        rc = prepare_pairs(hs, k, ws, P.data());
        if (rc) return rc;
    }
    if (ws.sep_cap == 0) {
        rc = ensure_sep_pool(h, ws, 2 * edge_cap + 1024, 0, st);
        if (rc) return rc;
    }
    {   // problem descriptors and vertex maps: uploaded only when they changed
        const size_t nk = (size_t)std::max(k, 1), nv = (size_t)std::max(total_vtx, 0);
        const size_t b0 = nk * sizeof(ProblemDev), b1 = nv * sizeof(int32_t), b2 = nk * sizeof(int32_t);
        const void* dst[3] = {ws.probs, ws.vtx_prob, ws.vtx_first};
        std::vector<uint8_t> blob(sizeof dst + b0 + b1 + b2);
        std::memcpy(blob.data(), dst, sizeof dst);
        std::memcpy(blob.data() + sizeof dst, P.data(), b0);
        std::memcpy(blob.data() + sizeof dst + b0, vtx_prob.data(), b1);
        std::memcpy(blob.data() + sizeof dst + b0 + b1, vtx_first.data(), b2);
        if (blob != ws.up_last) {
            if (blob.size() > ws.h_up_cap) {
                if (ws.h_up) cudaFreeHost(ws.h_up);
                ws.h_up = nullptr;
                ws.h_up_cap = 0;
                CK(cudaMallocHost((void**)&ws.h_up, blob.size()));
                ws.h_up_cap = blob.size();
            }
            // the staging buffer is free: every call ends with its stream drained
            std::memcpy(ws.h_up, blob.data(), blob.size());
            const uint8_t* src = ws.h_up + sizeof dst;
            CK(cudaMemcpyAsync(ws.probs, src, b0, cudaMemcpyHostToDevice, st));
            CK(cudaMemcpyAsync(ws.vtx_prob, src + b0, b1, cudaMemcpyHostToDevice, st));
            CK(cudaMemcpyAsync(ws.vtx_first, src + b0 + b1, b2, cudaMemcpyHostToDevice, st));
            ws.up_last.swap(blob);
        }
    }
    long long launches = 0;
    const bool persistent = *allow_loop && !shard && !plain && !gram && !nbr1 && h->opt.loop == FBN_LOOP_DEVICE &&
                            total_vtx <= kLoopVertices;
    const LoopShare share(h->device, persistent);   // until this call's work is done
    if (!gram && !persistent) {   // the complete graph (the Gram's decisions write every pair themselves)
        k_init_graph<<<total_vtx, 256, 0, st>>>(ws.probs, ws.vtx_prob, ws.vtx_first, total_vtx);
        CK(cudaGetLastError());
        launches = 1;
    }
    if (nbr1) {
        CK(launch_pack4(ws.probs, ws.vtx_prob, ws.vtx_first, total_vtx, st));
        launches += 1;
    }

    if (!ws.dev_sms) {
        int sms = 0;
        CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device));
        CK(set_kernel_smem(kWarpSmemBytes, kBigSmemBytes, kSmemBytes));
        // CTAs of the small-table pool (any group size) and of the big-table pool
        ws.grid_small = sms * std::max(1, pool_blocks_per_sm(kClassWarp, kWarpSmemBytes));
        ws.grid_big = sms * std::max(1, pool_blocks_per_sm(kClassCta, kBigSmemBytes));
        ws.grid_marg = sms * std::max(1, pool_blocks_per_sm(kClassMarg, 0));
        int per_sm = 0;
        CK(prepare_loop(kWarpSmemBytes, &per_sm));
        ws.grid_loop = sms * std::min(2, per_sm);
        ws.dev_sms = sms;
    }
    const int dev_sms = ws.dev_sms, grid_small = ws.grid_small, grid_big = ws.grid_big, grid_marg = ws.grid_marg;
    const long long groups[4] = {(long long)grid_small * 8, (long long)grid_small * 4, (long long)grid_small * 2,
                                 (long long)grid_small};
    const long long groups_big[4] = {grid_big, grid_big, grid_big, grid_big};   // whole CTAs
    const int grid_plain = 2 * dev_sms;
    double mean_n = 0;
    for (int p = 0; p < k; ++p) mean_n += (double)hs[p]->N / k;
    const int grid_aux = dev_sms * 4;   // grid-stride helpers (ordering, removal)
    // ranks per chunk: fixed by the option, else chosen on the device per depth
    const int gs_forced = plain ? 1 : h->opt.group_size;
    const long long gs_edges = 8LL * grid_small * 8;   // live edges from which 4 ranks per claim pay
    // G^2 with the declared df is decided from the n ln n table (pool form)
    long long max_N = 0;
    for (int p = 0; p < k; ++p) max_N = std::max<long long>(max_N, hs[p]->N);
    const bool use_lut = !plain && h->opt.statistic == FBN_STAT_G2 && h->opt.df_mode == FBN_DF_FIXED && max_N < kLutMaxN;
    if (use_lut && max_N + 1 > ws.lut_n) {
        dfree(ws.lut);
        ws.lut = nullptr;
        ws.lut_n = 0;
        CK(dalloc(&ws.lut, max_N + 1));
        ws.lut_n = max_N + 1;
        k_lut<<<(unsigned)((ws.lut_n + 255) / 256), 256, 0, st>>>(ws.lut, (int)ws.lut_n);
        CK(cudaGetLastError());
    }
    // an entry's error: two roundings of n ln n in FP64, one to the unit
    const double lut_top = (double)std::max<long long>(max_N, 2) * std::log((double)std::max<long long>(max_N, 2));
    const long long lut_err = (long long)(lut_top * 5e-16 * 68719476736.0) + 2;
    // largest table of the small class; the plain form runs every edge on a CTA
    const long long wcap = plain ? 0 : slice_cells((long long)(kWarpSmemBytes / 4), !use_lut);
    const int forced = h->opt.group_threads;
    if (ws.crit_alpha != alpha) {
        CK(cudaMemsetAsync(ws.crit_keys, 0, kCritCap * sizeof(long long), st));
        CK(cudaMemsetAsync(ws.crit_dense, 0, kCritDense * sizeof(double), st));
        CK(cudaMemsetAsync(ws.crit_dense_f, 0, kCritDense * sizeof(float2), st));
        CK(cudaMemsetAsync(ws.crit_dense_q, 0, kCritDense * sizeof(long long), st));
        ws.crit_alpha = alpha;
    }
    CritTableDev ct{ws.crit_keys, ws.crit_vals, kCritCap, kCritDense, ws.crit_dense, ws.crit_dense_f, ws.crit_dense_q};

    if (!persistent) {
        CK(cudaMemsetAsync(ws.d_rec, 0, kMaxDepthRecords * sizeof(DepthRecord), st));
        CK(cudaMemsetAsync(ws.hist, 0, 2 * ws.ord_cap * sizeof(unsigned long long), st));
        CK(cudaMemsetAsync(ws.cursor, 0, 2 * ws.ord_cap * sizeof(unsigned long long), st));
    }
    if (h->tune != ws.tune_loaded) {   // the autotuner's per-depth choices
        std::vector<int> t(kMaxDepthRecords, 0);
        for (size_t d = 0; d < h->tune.size() && d < t.size(); ++d) t[d] = h->tune[d];
        CK(cudaMemcpyAsync(ws.d_tune, t.data(), t.size() * sizeof(int), cudaMemcpyHostToDevice, st));
        ws.tune_loaded = h->tune;
    }
    DepthCounters c0{};
    c0.active = 1;
    c0.tune = h->tune.empty() ? nullptr : ws.d_tune;
    c0.rec = ws.d_rec;
    *ws.h_ctr = c0;
    if (!persistent) CK(cudaMemcpyAsync(ws.d_ctr, ws.h_ctr, sizeof(DepthCounters), cudaMemcpyHostToDevice, st));

    PoolArgs base{};
    base.probs = ws.probs;
    base.edges = ws.edges;
    base.min_accept = ws.min_accept;
    base.edge_cap = ws.edge_cap;
    base.sorted = ws.sorted;
    base.ctr = ws.d_ctr;
    base.binom = ws.binom;
    base.binom_rows = ws.brows;
    base.crit = ct;
    base.alpha = alpha;
    base.stat = h->opt.statistic;
    base.df_mode = h->opt.df_mode;
    base.split_tab = ws.split_tab;
    base.split_ticket = ws.split_ticket;
    base.split_stride = kSplitStride;
    base.lut = use_lut ? ws.lut : nullptr;
    base.lut_err = lut_err;

    if (ws.split_dirty) {
        CK(cudaMemsetAsync(ws.split_tab, 0, kSplitItems * kSplitStride * sizeof(int), st));
        CK(cudaMemsetAsync(ws.split_ticket, 0, kSplitItems * sizeof(unsigned), st));
    }
    ws.split_dirty = true;   // until this call completes its loop

    // The kernels of one depth after the edge list: ordering and the pool of
    // each class; then removal and the end of the depth.
    auto enqueue_order = [&](bool marg) {   // both classes up front: their sorted orders do not overlap
        ScanClass sc[2];
        for (int cls = 0; cls < 2; ++cls) {
            sc[cls].hist = ws.hist + cls * ws.ord_cap;
            sc[cls].alive = ws.alive + cls * ws.ord_cap;
            sc[cls].base = ws.base + cls * ws.ord_cap;
            for (int k = 0; k < 4; ++k) sc[cls].groups[k] = cls == 0 ? groups[k] : groups_big[k];
            sc[cls].smem_ints = (long long)((cls == 0 ? kWarpSmemBytes : kBigSmemBytes) / 4);
            sc[cls].mid_ints = (long long)(kSmemBytes / 4);
        }
        launch_order(ws.probs, ws.edges, ws.edge_cap, marg ? 1 : 2, ws.d_ctr, sc, ws.cursor, ws.cursor + ws.ord_cap,
                     ws.sorted, mean_n, forced, kSplitStride, 1, marg, !use_lut, grid_aux, st);
    };
    auto enqueue_tests = [&]() {
        const int nclass = 2;
        if (!plain) enqueue_order(false);
        for (int cls = 0; cls < nclass; ++cls) {
            PoolArgs a = base;
            a.cls = cls;
            const bool small = cls == kClassWarp && !plain;
            const size_t smem = small ? kWarpSmemBytes : plain ? kSmemBytes : kBigSmemBytes;
            a.smem_ints = (int)(smem / 4);
            if (!small && ws.gs_cells > 0) {
                a.gscratch = ws.gscratch;
                a.gscratch_ints = 3 * ws.gs_cells + 64;
            }
            if (plain) {
                launch_plain(a, grid_plain, kSmemBytes, st);
                continue;
            }
            a.base = ws.base + cls * ws.ord_cap;
            a.sorted = ws.sorted;
            launch_pool(a, cls, small ? grid_small : grid_big, smem, st);
            if (!small && !use_lut) {   // one of the two runs (choose_pool)
                a.smem_ints = (int)(kSmemBytes / 4);
                launch_pool_mid(a, grid_plain, kSmemBytes, st);
            }
        }
    };
    // depth 1 from one-hot planes: every edge is in the small-table class
    auto enqueue_marg = [&]() {
        enqueue_order(true);
        PoolArgs a = base;
        a.cls = kClassWarp;
        a.base = ws.base;
        a.sorted = ws.sorted;
        launch_pool_marg(a, grid_marg, st);
    };
    auto enqueue_popc0 = [&]() {
        const long long tasks = (long long)total_vtx * max_n;
        launch_pairs_popc(ws.probs, ws.vtx_prob, ws.vtx_first, total_vtx, max_n, shard ? ws.d_owned : nullptr, base,
                          (int)std::min<long long>((tasks + 7) / 8, dev_sms * 8), st);
    };
    auto enqueue_head = [&](bool marg = false) {
        launch_snapshot(ws.probs, ws.vtx_prob, ws.vtx_first, total_vtx, ws.d_ctr, st);
        launch_edges(ws.probs, ws.vtx_prob, ws.vtx_first, total_vtx, gs_forced, gs_edges, ws.binom, ws.brows, wcap,
                     marg ? (long long)(kMargThreads / 32) * grid_marg : 0, shard ? ws.d_owned : nullptr, ws.edges, ws.min_accept, ws.edge_cap, ws.d_ctr,
                     ws.hist, st);
    };
    auto enqueue_tail = [&]() {
        launch_apply(ws.probs, ws.edges, ws.min_accept, ws.edge_cap, ws.binom, ws.sep_pool, ws.sep_cap, ws.d_ctr,
                     grid_aux, st);
        launch_depth_end(ws.d_ctr, ws.d_rec, max_depth, ws.hist, ws.cursor, st);
    };
    const int body_launches = plain ? 7 : use_lut ? 9 : 10;
    auto capture_loop = [&]() -> cudaError_t {
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaGraphCreate(&g, 0);
        if (e != cudaSuccess) return e;
        auto give_up = [&](cudaError_t err) {
            cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
            if (cudaStreamIsCapturing(st, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone) {
                cudaGraph_t tmp = nullptr;
                cudaStreamEndCapture(st, &tmp);
            }
            cudaGetLastError();
            cudaGraphDestroy(g);
            return err;
        };
        cudaGraphConditionalHandle cond{};
        if ((e = cudaGraphConditionalHandleCreate(&cond, g, 0, 0)) != cudaSuccess) return give_up(e);
        // top level: the first depth's edge list and the loop condition
        if ((e = cudaStreamBeginCaptureToGraph(st, g, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal)) !=
            cudaSuccess)
            return give_up(e);
        enqueue_head();
        launch_gate(ws.d_ctr, cond, st);
        cudaGraphNode_t gate_node = nullptr;
        {
            cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
            const cudaGraphNode_t* deps = nullptr;
            size_t nd = 0;
            if ((e = cudaStreamGetCaptureInfo(st, &cs, nullptr, nullptr, &deps, nullptr, &nd)) != cudaSuccess)
                return give_up(e);
            if (cs != cudaStreamCaptureStatusActive || nd != 1) return give_up(cudaErrorStreamCaptureInvalidated);
            gate_node = deps[0];
        }
        cudaGraph_t out = nullptr;
        if ((e = cudaStreamEndCapture(st, &out)) != cudaSuccess) return give_up(e);
        // the while node and its body: one depth, then the next one's edge list
        cudaGraphNodeParams cp{};
        cp.type = cudaGraphNodeTypeConditional;
        cp.conditional.handle = cond;
        cp.conditional.type = cudaGraphCondTypeWhile;
        cp.conditional.size = 1;
        cudaGraphNode_t cn = nullptr;
        if ((e = cudaGraphAddNode(&cn, g, &gate_node, nullptr, 1, &cp)) != cudaSuccess) return give_up(e);
        cudaGraph_t body = cp.conditional.phGraph_out[0];
        if ((e = cudaStreamBeginCaptureToGraph(st, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal)) !=
            cudaSuccess)
            return give_up(e);
        enqueue_tests();
        enqueue_tail();
        enqueue_head();
        launch_gate(ws.d_ctr, cond, st);
        if ((e = cudaStreamEndCapture(st, &out)) != cudaSuccess) return give_up(e);
        e = cudaGraphInstantiate(&ws.loop, g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) {
            ws.loop = nullptr;
            cudaGetLastError();
        }
        return e;
    };

    // The generic depths as one graph: the edge list of the first one, then a
    // device-driven while loop whose body tests a depth, removes its edges,
    // ends it and lists the next depth's edges (k_gate: go on or stop).
    // Captured once per configuration: every argument it holds is in the key.
    auto ensure_graph = [&]() -> int {
        std::vector<uint8_t> key;
        auto put = [&](const void* p, size_t n) {
            const uint8_t* b = (const uint8_t*)p;
            key.insert(key.end(), b, b + n);
        };
        const void* ptrs[] = {ws.probs, ws.vtx_prob, ws.vtx_first, ws.binom, ws.edges, ws.min_accept, ws.d_ctr,
                              ws.hist, ws.alive, ws.base, ws.cursor, ws.sorted, ws.gscratch, ws.sep_pool, ws.d_rec,
                              ws.crit_keys, ws.crit_vals, ws.crit_dense, ws.crit_dense_f, ws.crit_dense_q, ws.lut,
                              ws.split_tab, ws.split_ticket};
        put(ptrs, sizeof ptrs);
        const long long ints[] = {total_vtx, gs_forced, gs_edges, ws.brows, wcap, ws.edge_cap, ws.ord_cap, forced,
                                  grid_aux, grid_small, grid_big, ws.gs_cells, ws.sep_cap, max_depth, plain,
                                  h->opt.statistic, h->opt.df_mode, use_lut, lut_err,
                                  groups[0], groups[1], groups[2], groups[3]};
        put(ints, sizeof ints);
        put(&mean_n, sizeof mean_n);
        put(&alpha, sizeof alpha);
        if (key != ws.graph_key) {
            if (ws.loop) cudaGraphExecDestroy(ws.loop);
            ws.loop = nullptr;
            ws.graph_key.clear();
            // with programmatic launches first, else without (bodies of
            // conditional nodes may refuse programmatic edges)
            cudaError_t err = cudaSuccess;
            for (int pdl = 1; pdl >= 0 && !ws.loop; --pdl) {
                set_pdl(pdl != 0);
                err = capture_loop();
            }
            set_pdl(true);
            if (!ws.loop) return fail(h, FBN_ECUDA, "depth loop graph: %s", cudaGetErrorString(err));
            ws.graph_key = key;
        }
        return FBN_OK;
    };
    if (!shard && !persistent && (rc = ensure_graph())) return rc;

    fbn_stats stats{};
    int d_loop = 0;   // first depth of the graph loop
    bool direct_out = persistent && k == 1;
    const long long* h_tot = nullptr;
    if (persistent) {
        LoopArgs la{};
        la.probs = ws.probs;
        la.vtx_prob = ws.vtx_prob;
        la.vtx_first = ws.vtx_first;
        la.total_vertices = total_vtx;
        la.max_n = max_n;
        la.gs_forced = gs_forced;
        la.gs_edges = gs_edges;
        la.binom = ws.binom;
        la.brows = ws.brows;
        la.warp_cells_cap = wcap;
        la.edges = ws.edges;
        la.min_accept = ws.min_accept;
        la.edge_cap = ws.edge_cap;
        la.ctr = ws.d_ctr;
        la.hist = ws.hist;
        la.cursor = ws.cursor;
        la.ord_cap = ws.ord_cap;
        const int grid = share.grid(total_vtx <= kLoopOneCta ? dev_sms : ws.grid_loop, dev_sms);
        for (int cls = 0; cls < 2; ++cls) {
            la.sc[cls].hist = ws.hist + cls * ws.ord_cap;
            la.sc[cls].alive = ws.alive + cls * ws.ord_cap;
            la.sc[cls].base = ws.base + cls * ws.ord_cap;
            for (int q = 0; q < 4; ++q) la.sc[cls].groups[q] = cls == 0 ? ((long long)grid * 8) >> q : grid;
            la.sc[cls].smem_ints = (long long)(kWarpSmemBytes / 4);
        }
        la.sorted = ws.sorted;
        la.mean_n = mean_n;
        la.forced_group = forced;
        la.split_stride = kSplitStride;
        la.need_marg = !use_lut;
        la.sep_pool = ws.sep_pool;
        la.sep_cap = ws.sep_cap;
        la.rec = ws.d_rec;
        la.max_depth = max_depth;
        la.popc0 = popc0;
        la.marg1 = marg1;
        la.small = base;
        la.small.cls = kClassWarp;
        la.small.smem_ints = (int)(kWarpSmemBytes / 4);
        la.small.base = ws.base;
        la.big = la.small;
        la.big.cls = kClassCta;
        la.big.base = ws.base + ws.ord_cap;
        la.small.hand_over = la.big.hand_over = 1;
        // 2^23 polls are seconds
        la.spin_limit = h->opt.wait_limit < 0 ? 0u : h->opt.wait_limit > 0 ? (unsigned)h->opt.wait_limit : 1u << 23;
        if (!ws.d_bar) {
            CK(dalloc(&ws.d_bar, 2));
            CK(cudaMemsetAsync(ws.d_bar, 0, 2 * sizeof(unsigned), st));
        }
        if (!ws.h_left) CK(cudaMallocHost((void**)&ws.h_left, sizeof(unsigned)));
        CK(cudaHostGetDevicePointer((void**)&la.left, ws.h_left, 0));
        *ws.h_left = 0;
        la.bar = ws.d_bar;
        if (k == 1 && h->n <= kTurnVertices) {
            if (!ws.d_bits) CK(dalloc(&ws.d_bits, kTurnVertices * (kTurnVertices / 32)));
            la.bits = ws.d_bits;
        }
        la.init = c0;
        if (direct_out) {   // one problem: every result straight to the host
            const long long R = edge_cap;
            CK(grow_pinned(&ws.h_adj, &ws.h_adj_cap, ((size_t)h->n * h->n + 15) / 16 * 16));
            const size_t csr = CsrPlace::bytes(R, ws.sep_cap);
            CK(acquire_stage(ws, csr + 16));
            if (!h->d_sep_cnt) CK(dalloc(&h->d_sep_cnt, 2 * (size_t)h->n));
            CK(cudaHostGetDevicePointer((void**)&la.h_ctr, ws.h_ctr, 0));
            CK(cudaHostGetDevicePointer((void**)&la.h_rec, ws.h_rec, 0));
            if (adj_out && adj_out[0]) CK(cudaHostGetDevicePointer((void**)&la.h_adj, ws.h_adj, 0));
            const CsrPlace at(0, R);
            la.h_pairs = reinterpret_cast<int32_t*>(ws.stage->dev + at.pairs);
            la.h_offs = reinterpret_cast<int64_t*>(ws.stage->dev + at.offs);
            la.h_members = reinterpret_cast<int32_t*>(ws.stage->dev + at.members);
            la.h_tot = reinterpret_cast<long long*>(ws.stage->dev + csr);
            h_tot = reinterpret_cast<const long long*>(ws.stage->p + csr);
            la.sep_cnt = h->d_sep_cnt;
        }
        CK(launch_loop(la, grid, kWarpSmemBytes, st));
        launches += 1;
    }
    bool direct1 = false;   // depth 1 as the neighbourhood product (timed by events)
    if (shard || persistent) {
        // depth by depth below; one kernel above
    } else if (gram) {
        rc = run_gram(h, ws, k, total_vtx, &ws.d_ctr->status, ws.d_ctr, ws.kev[2 * FBN_MAX_DEPTHS],
                      ws.kev[2 * FBN_MAX_DEPTHS + 1]);
        if (rc) return rc;
        PairsGramArgs pa;
        pa.emit = marg1;
        pa.total_pairs = edge_cap;
        pa.crit = ct;
        pa.alpha = alpha;
        pa.ctr = ws.d_ctr;
        pa.stat = h->opt.statistic;
        pa.df_mode = h->opt.df_mode;
        for (int p = 0; p < k; ++p) pa.max_arity = std::max(pa.max_arity, hs[p]->max_arity);
        CK(launch_pairs_gram(ws.probs, ws.vtx_prob, ws.vtx_first, total_vtx, max_n, pa, dev_sms, st));
        launch_depth_end(ws.d_ctr, ws.d_rec, max_depth, ws.hist, ws.cursor, st);
        launches += pa.max_arity > kWideArity ? 5 : 4;
        d_loop = 1;
    } else if (popc0) {
        enqueue_head();
        enqueue_popc0();
        enqueue_tail();
        launches += 5;
        d_loop = 1;
    }
    if (marg1 && !shard && !persistent) {
        enqueue_head(true);
        enqueue_marg();
        enqueue_tail();
        launches += 7;
        d_loop = 2;
    }
    if (nbr1 && (max_depth < 0 || max_depth >= 1)) {
        if (d_loop == 0) {   // depth 0 on the pool, launched directly
            enqueue_head();
            enqueue_tests();
            enqueue_tail();
            launches += body_launches - 1;
        }
        enqueue_head();
        CK(cudaEventRecord(ws.tev[0], st));
        CK(launch_nbr1(ws.probs, ws.vtx_prob, ws.vtx_first, total_vtx, ws.edges, ws.min_accept, ct, alpha, ws.d_ctr,
                       dev_sms, h->opt.wait_limit, st));
        CK(cudaEventRecord(ws.tev[1], st));
        enqueue_tail();
        launches += 5;
        direct1 = true;
        d_loop = 2;
    }
    bool loop = !persistent && (max_depth < 0 || d_loop <= max_depth);
    const bool host_loop = h->opt.loop == FBN_LOOP_HOST || shard;
    if (shard) {
        // Several processes learn this skeleton together (Section IV-A's
        // edge-level partition across devices): every process holds the same
        // graph; per depth, the caller's `own` picks this process's edges, the
        // process tests them and exports its removals as (i, j, rank) records,
        // the caller's `exchange` gathers every process's records, and each
        // process applies all of them to the same snapshot.  The host decides
        // the stop, from the graph every process shares.
        const int n = h->n;
        std::vector<uint8_t> adj_h((size_t)n * n), own_h((size_t)n * n);
        std::vector<int64_t> local, all;
        for (int d = 0;; ++d) {
            if (max_depth >= 0 && d > max_depth) break;
            if (d >= kMaxDepthRecords - 1 || d > kMaxD) break;
            CK(cudaMemcpyAsync(adj_h.data(), h->d_adj, adj_h.size(), cudaMemcpyDeviceToHost, st));
            CK(cudaStreamSynchronize(st));
            std::vector<int> deg(n, 0);
            for (int i = 0; i < n; ++i)
                for (int j = 0; j < n; ++j) deg[i] += adj_h[(size_t)i * n + j] != 0;
            bool any = false;   // an edge with a side of at least d candidates
            for (int i = 0; i < n && !any; ++i)
                for (int j = i + 1; j < n && !any; ++j)
                    any = adj_h[(size_t)i * n + j] && std::max(deg[i], deg[j]) - 1 >= d;
            if (!any) break;
            std::fill(own_h.begin(), own_h.end(), 0);
            if (shard->own(shard->ctx, d, n, adj_h.data(), own_h.data()) != 0)
                return fail(h, FBN_EINVAL, "the own callback failed at depth %d", d);
            CK(cudaMemcpyAsync(ws.d_owned, own_h.data(), own_h.size(), cudaMemcpyHostToDevice, st));
            CK(cudaMemsetAsync(ws.d_shard_count, 0, sizeof(unsigned long long), st));
            enqueue_head(d == 1 && marg1);
            if (d == 0 && popc0) enqueue_popc0();
            else if (d == 1 && marg1) enqueue_marg();
            else enqueue_tests();
            launch_shard_export(ws.probs, ws.edges, ws.min_accept, ws.edge_cap, ws.d_ctr, ws.d_shard, ws.d_shard_count,
                                grid_aux, st);
            unsigned long long m = 0;
            CK(cudaMemcpyAsync(&m, ws.d_shard_count, sizeof m, cudaMemcpyDeviceToHost, st));
            CK(cudaStreamSynchronize(st));
            if ((long long)m > ws.shard_cap) return fail(h, FBN_ECUDA, "removal records over their bound");
            local.resize(3 * m);
            if (m) CK(cudaMemcpy(local.data(), ws.d_shard, 3 * m * sizeof(int64_t), cudaMemcpyDeviceToHost));
            const long long cap = (long long)n * (n - 1) / 2;
            all.assign(3 * (size_t)cap, 0);
            int64_t n_all = 0;
            if (shard->exchange(shard->ctx, d, local.data(), (int64_t)m, all.data(), cap, &n_all) != 0 || n_all < 0 ||
                n_all > cap)
                return fail(h, FBN_EINVAL, "the exchange callback failed at depth %d", d);
            // every record must name an edge of the shared graph once, with a
            // rank inside its rank space (checked here: the kernel trusts them)
            std::vector<uint8_t> seen((size_t)n * n, 0);
            for (long long t = 0; t < n_all; ++t) {
                const long long i = (long long)all[3 * t], j = (long long)all[3 * t + 1], r = (long long)all[3 * t + 2];
                if (i < 0 || j <= i || j >= n || !adj_h[(size_t)i * n + j] || seen[(size_t)i * n + j] || r < 0)
                    return fail(h, FBN_EINVAL, "bad removal record (%lld, %lld, %lld) at depth %d", i, j, r, d);
                seen[(size_t)i * n + j] = 1;
                if (d > 0) {
                    double ti = 1, tj = 1;   // C(deg - 1, d) on each side, in double (no overflow to care about here)
                    for (int q = 0; q < d; ++q) {
                        ti = ti * (deg[i] - 1 - q) / (q + 1);
                        tj = tj * (deg[j] - 1 - q) / (q + 1);
                    }
                    if ((double)r >= std::max(ti, 0.0) + std::max(tj, 0.0))
                        return fail(h, FBN_EINVAL, "removal record rank %lld out of range at depth %d", r, d);
                } else if (r != 0) {
                    return fail(h, FBN_EINVAL, "removal record rank %lld out of range at depth 0", r);
                }
            }
            if (n_all) CK(cudaMemcpyAsync(ws.d_shard, all.data(), 3 * n_all * sizeof(int64_t), cudaMemcpyHostToDevice, st));
            launch_shard_apply(ws.probs, ws.d_shard, n_all, ws.binom, ws.brows, ws.sep_pool, ws.sep_cap, ws.d_ctr,
                               grid_aux, st);
            launch_depth_end(ws.d_ctr, ws.d_rec, -1, ws.hist, ws.cursor, st);
            launch_shard_continue(ws.d_ctr, st);
            launches += body_launches + 1;
        }
    } else if (loop && host_loop) {
        // the same kernels, depth by depth: the edge list, then while the
        // depth has an edge to test, its tests, removal and end, and the next
        // depth's edge list
        enqueue_head();
        launches += 2;
        for (;;) {
            CK(cudaMemcpyAsync(ws.h_ctr, ws.d_ctr, sizeof(DepthCounters), cudaMemcpyDeviceToHost, st));
            CK(cudaStreamSynchronize(st));
            if (!ws.h_ctr->active || ws.h_ctr->n_edges[0] + ws.h_ctr->n_edges[1] == 0) break;
            enqueue_tests();
            enqueue_tail();
            enqueue_head();
        }
    } else if (loop) {
        CK(cudaGraphLaunch(ws.loop, st));
        launches += 3;
    }
    CK(cudaGetLastError());
    // The counters and the graphs to the host, with the call's synchronisation.
    bool adj_staged = false;   // the adjacency comes from the pinned staging after the synchronisation
    std::vector<int> staged;
    std::vector<size_t> staged_at;
    auto fetch = [&]() -> int {
        adj_staged = false;
        if (direct_out) {
            if (adj_out && adj_out[0]) {
                cudaPointerAttributes attr{};
                const cudaError_t pe = cudaPointerGetAttributes(&attr, adj_out[0]);
                cudaGetLastError();
                adj_staged = pe != cudaSuccess || attr.type == cudaMemoryTypeUnregistered || attr.type == cudaMemoryTypeHost;
            }
        } else {
            CK(cudaMemcpyAsync(ws.h_ctr, ws.d_ctr, sizeof(DepthCounters), cudaMemcpyDeviceToHost, st));
            CK(cudaMemcpyAsync(ws.h_rec, ws.d_rec, kMaxDepthRecords * sizeof(DepthRecord), cudaMemcpyDeviceToHost, st));
        }
        // The graphs go out with the counters (dropped if the call is retried): a
        // batch's for pageable memory through one pinned buffer of at most
        // kAdjStageBytes, the others and what is over that by a copy each.  (One
        // graph of 1,000 variables takes as long either way.)
        staged.clear();
        staged_at.clear();
        if (adj_out && !adj_staged) {
            size_t total = 0;
            for (int p = 0; p < k; ++p) {
                if (!adj_out[p]) continue;
                const size_t nn = (size_t)hs[p]->n * hs[p]->n, padded = (nn + 15) / 16 * 16;
                cudaPointerAttributes attr{};
                const cudaError_t pe = cudaPointerGetAttributes(&attr, adj_out[p]);
                cudaGetLastError();
                if (k > 1 && (pe != cudaSuccess || attr.type == cudaMemoryTypeUnregistered) && total + padded <= kAdjStageBytes) {
                    staged.push_back(p);
                    staged_at.push_back(total);
                    total += padded;
                } else {
                    CK(cudaMemcpyAsync(adj_out[p], hs[p]->d_adj, nn, cudaMemcpyDefault, st));
                }
            }
            if (total) {
                CK(grow_pinned(&ws.h_adj, &ws.h_adj_cap, total));
                uint4* dst = nullptr;
                CK(cudaHostGetDevicePointer((void**)&dst, ws.h_adj, 0));
                for (size_t s0 = 0; s0 < staged.size(); s0 += kAdjJob) {
                    const int m = (int)std::min<size_t>(kAdjJob, staged.size() - s0);
                    AdjJob job{};
                    long long most = 1;
                    for (int q = 0; q < m; ++q) {
                        const fbn_handle* g = hs[staged[s0 + q]];
                        job.src[q] = g->d_adj;
                        job.words[q] = ((long long)g->n * g->n + 15) / 16;
                        job.off[q] = (long long)(staged_at[s0 + q] / 16);
                        most = std::max(most, job.words[q]);
                    }
                    k_adj_out<<<dim3((unsigned)std::min<long long>((most + 1023) / 1024, 1024), m), 256, 0, st>>>(job, dst);
                    CK(cudaGetLastError());
                    launches += 1;
                }
            }
        }
        CK(cudaStreamSynchronize(st));
        return FBN_OK;
    };
    if ((rc = fetch())) return rc;
    if (persistent && *ws.h_left == kLoopGaveUp) {   // the barrier's words and the counters are not whole
        CK(cudaMemsetAsync(ws.d_bar, 0, 2 * sizeof(unsigned), st));
        CK(cudaStreamSynchronize(st));
        *allow_loop = false;
        *retry = true;
        return FBN_OK;
    }
    if (persistent && *ws.h_left >= kLoopHandedOver) {   // the depths from there on as a graph
        d_loop = (int)((*ws.h_left & (kLoopSplit - 1)) - kLoopHandedOver);
        direct_out = false;
        loop = true;
        if ((rc = ensure_graph())) return rc;
        if (*ws.h_left & kLoopSplit) {
            CK(cudaMemsetAsync(ws.split_tab, 0, kSplitItems * kSplitStride * sizeof(int), st));
            CK(cudaMemsetAsync(ws.split_ticket, 0, kSplitItems * sizeof(unsigned), st));
        }
        CK(cudaGraphLaunch(ws.loop, st));
        launches += 3;
        if ((rc = fetch())) return rc;
    }
    if (adj_staged) std::memcpy(adj_out[0], ws.h_adj, (size_t)h->n * h->n);
    for (size_t s = 0; s < staged.size(); ++s)
        std::memcpy(adj_out[staged[s]], ws.h_adj + staged_at[s], (size_t)hs[staged[s]]->n * hs[staged[s]]->n);
    if (loop && !shard) launches += (long long)(body_launches - (host_loop ? 1 : 0)) * std::max(0, ws.h_ctr->d - d_loop);
    if (direct1) {
        float kms = 0.f;
        CK(cudaEventElapsedTime(&kms, ws.tev[0], ws.tev[1]));
        stats.test_ms[1] = kms;
    }
    const DepthCounters& c = *ws.h_ctr;
    if (c.status == 0) ws.split_dirty = false;   // every split test's last part zeroed its table
    if (c.status & (kStatusSepPool | kStatusScratch)) {
        if (c.status & kStatusSepPool) {
            rc = ensure_sep_pool(h, ws, 2 * ws.sep_cap + 2 * (long long)c.sep_used, 0, st);
            if (rc) return rc;
        }
        if (c.status & kStatusScratch) {
            if (c.need_cells <= 0 || c.need_cells > kMaxCells) return check_status(h, kStatusTooBig);
            ws.gs_cells = std::max<long long>(2 * ws.gs_cells, c.need_cells);
            rc = ensure_gscratch(h, ws, (3 * ws.gs_cells + 64) * std::max(grid_big, grid_plain));
            if (rc) return rc;
        }
        *retry = true;
        return FBN_OK;
    }
    rc = check_status(h, c.status);
    if (rc) return rc;

    for (int d = 0; d < kMaxDepthRecords; ++d) {
        const DepthRecord& r = ws.h_rec[d];
        if (r.edges == 0) break;   // the depth that found no edge: Algorithm 1 stopped before it
        if (d >= FBN_MAX_DEPTHS) break;
        stats.depths = d + 1;
        stats.edges[d] = r.edges;
        stats.tests[d] = r.tests;
        stats.tests_oracle[d] = r.tests_oracle;
        stats.test_samples[d] = r.test_samples;
        stats.popc_work[d] = r.popc_work;
        stats.smem_updates[d] = r.smem_updates;
        stats.removed[d] = r.removed;
        const unsigned long long next = d + 1 < kMaxDepthRecords ? ws.h_rec[d + 1].t_begin : 0;
        const unsigned long long end = next > r.t_begin ? next : r.t_end;
        stats.ms[d] = end > r.t_begin && r.t_begin ? (float)((end - r.t_begin) * 1e-6) : 0.f;
        if (!(direct1 && d == 1) && r.t_tests_end > r.t_tests && r.t_tests)
            stats.test_ms[d] = (float)((r.t_tests_end - r.t_tests) * 1e-6);
    }
    if (gram) {
        float gms = 0.f;
        CK(cudaEventElapsedTime(&gms, ws.kev[2 * FBN_MAX_DEPTHS], ws.kev[2 * FBN_MAX_DEPTHS + 1]));
        stats.gram_ms = gms;
        for (int p = 0; p < k; ++p) {
            stats.gram_rows += hs[p]->M - hs[p]->n;
            stats.gram_samples = std::max<int64_t>(stats.gram_samples, hs[p]->K);
        }
    }
    stats.launches = launches;
    // every problem's sets stay on the device until asked for; a batch's
    // members live in the first handle's pool, which its next call reuses, so
    // the batch keeps a device copy of the used part
    std::shared_ptr<DeviceInts> snap;
    if (k > 1) {
        snap = std::make_shared<DeviceInts>();
        snap->n = std::max<long long>(1, (long long)c.sep_used);
        CK(dalloc(&snap->d, snap->n));
        if (c.sep_used)
            CK(cudaMemcpyAsync(snap->d, ws.sep_pool, c.sep_used * sizeof(int32_t), cudaMemcpyDeviceToDevice, st));
        CK(cudaEventCreateWithFlags(&snap->ready, cudaEventDisableTiming));
        CK(cudaEventRecord(snap->ready, st));
    }
    for (int p = 0; p < k; ++p) {
        hs[p]->stats = stats;
        hs[p]->learnt = true;
        hs[p]->sep_pending = true;
        hs[p]->sep_pool_used = c.sep_used;
        set_snapshot(hs[p], snap);
    }
    if (direct_out) take_csr(h, ws.stage, CsrPlace(0, edge_cap), h_tot[0], h_tot[1]);   // already on the host
    return FBN_OK;
}

int run_skeleton(fbn_handle* const* hs, int k, double alpha, int32_t max_depth, uint8_t* const* adj_out = nullptr,
                 const ShardHooks* shard = nullptr)
{
    for (int p = 0; p < k; ++p) drop_sepsets(hs[p]);   // their pinned memory is written again
    bool allow_loop = true;
    for (int attempt = 0; attempt < 7; ++attempt) {
        bool retry = false;
        const int rc = run_skeleton_once(hs, k, alpha, max_depth, &retry, &allow_loop, adj_out, shard);
        if (rc || !retry) return rc;
    }
    return fail(hs[0], FBN_ENOMEM, "scratch or separating-set pool kept overflowing");
}

int check_test_args(fbn_handle* h, int32_t x, int32_t y, const int32_t* z, int32_t nz, long long* cells)
{
    if (!h) return FBN_EINVAL;
    if (x < 0 || x >= h->n || y < 0 || y >= h->n || x == y)
        return fail(h, FBN_EINVAL, "bad x=%d y=%d for n=%d", x, y, h->n);
    if (nz < 0 || nz > kMaxD || (nz > 0 && !z))
        return fail(h, FBN_EINVAL, "conditioning set size %d outside [0, %d]", nz, kMaxD);
    long long c = (long long)h->h_ar[x] * h->h_ar[y];
    for (int k = 0; k < nz; ++k) {
        if (z[k] < 0 || z[k] >= h->n || z[k] == x || z[k] == y)
            return fail(h, FBN_EINVAL, "bad conditioning variable %d", z[k]);
        for (int l = 0; l < k; ++l)
            if (z[l] == z[k]) return fail(h, FBN_EINVAL, "conditioning variable %d repeated", z[k]);
        c *= h->h_ar[z[k]];
        if (c > kMaxCells) return fail(h, FBN_ETOOBIG, "table exceeds %lld cells", kMaxCells);
    }
    *cells = c;
    return FBN_OK;
}

constexpr long long kCiHostTable = 1 << 16;   // cells of a table the kernel writes into pinned host memory

// One explicit test: its statistic, df and p into h->h_ci_out, or its table
// (want_table) into *table: pinned host memory, or h->d_table for large ones.
// One launch and one synchronisation: the descriptor goes by value and the
// results are written straight to the host (with copies each way a test of
// 5,000 samples took 48 us, of which the kernel was a quarter).
int run_ci(fbn_handle* h, int32_t x, int32_t y, const int32_t* z, int32_t nz, long long cells, bool want_table)
{
    CK(cudaSetDevice(h->device));
    cudaStream_t st = h->stream;
    if (!h->ci_cluster_max) CK(prepare_ci(kSmemBytes, &h->ci_cluster_max));
    CiArgs q{};
    for (int k = 0; k < nz + 2; ++k) {
        const int v = k < nz ? z[k] : k == nz ? x : y;
        q.rows[k] = h->d_data + (long long)v * h->ld;
        q.rad[k] = h->h_ar[v];
    }
    q.nrows = nz + 2;
    q.rx = h->h_ar[x];
    q.ry = h->h_ar[y];
    q.N = (int)h->N;
    q.cells = cells;
    q.smem_ints = (int)(kSmemBytes / 4);
    q.stat = h->opt.statistic;
    q.df_mode = h->opt.df_mode;
    const int k = ci_cluster(h->N, cells, h->ci_cluster_max);
    if (want_table) {
        if (cells <= kCiHostTable) {
            if (cells > h->h_table_cap) {
                if (h->h_table) cudaFreeHost(h->h_table);
                h->h_table = nullptr;
                h->h_table_cap = 0;
                CK(cudaMallocHost((void**)&h->h_table, cells * sizeof(int32_t)));
                h->h_table_cap = cells;
            }
            CK(cudaHostGetDevicePointer((void**)&q.table_out, h->h_table, 0));
        } else {
            if (cells > h->table_cap) {
                dfree(h->d_table);
                h->d_table = nullptr;
                h->table_cap = 0;
                CK(dalloc(&h->d_table, cells));
                h->table_cap = cells;
            }
            q.table_out = h->d_table;
        }
    } else {
        q.out = h->ci_out_dev;
        q.status = h->status_dev;
        q.lgamma_a = ci_lgamma(q.rx, q.ry, cells);
    }
    if (!ci_fits_smem(cells, q.rx, q.ry, k, q.smem_ints)) {
        const long long gints = 3 * cells + 64;
        if (gints > h->gscratch_ints) {
            dfree(h->d_gscratch);
            h->d_gscratch = nullptr;
            h->gscratch_ints = 0;
            CK(dalloc(&h->d_gscratch, gints));
            h->gscratch_ints = gints;
        }
        q.gtab = h->d_gscratch;
    }
    *h->h_status = 0;
    CK(launch_ci(q, k, kSmemBytes, st));
    CK(cudaStreamSynchronize(st));
    return check_status(h, *h->h_status);
}

// ---- autotuning --------------------------------------------------------
struct TuneChoice {
    std::vector<int> table;   // per-depth codes (empty: the fixed rules won)
    int depth0 = 0;
    fbn_tuning report{};
};
std::mutex g_tune_mu;
std::map<std::vector<long long>, TuneChoice> g_tune_cache;

// The workload shape a tuning applies to: device, options that shape the
// work, alpha, max depth, and every problem's (n, N, largest arity).
std::vector<long long> tune_key(fbn_handle* const* hs, int k, double alpha, int32_t max_depth)
{
    const fbn_handle* h = hs[0];
    long long abits = 0;
    std::memcpy(&abits, &alpha, sizeof abits);
    std::vector<long long> key = {h->device, k, h->opt.form, h->opt.statistic, h->opt.df_mode, h->opt.count,
                                  h->opt.group_threads, h->opt.depth0, h->opt.depth1, abits, max_depth};
    for (int p = 0; p < k; ++p) {
        key.push_back(hs[p]->n);
        key.push_back(hs[p]->N);
        key.push_back(hs[p]->max_arity);
    }
    return key;
}

void apply_tuning(fbn_handle* const* hs, int k, const std::vector<int>& table, int depth0)
{
    for (int p = 0; p < k; ++p) {
        hs[p]->tune = table;
        hs[p]->tune_depth0 = depth0;
    }
}

// Timed skeletons of the batch under a configuration: a first run warms
// (capture, lazily filled tables), then `reps` runs are timed with events on
// the stream; the whole time and every depth's test window (device clock) are
// the medians over the runs.
int timed_run(fbn_handle* const* hs, int k, double alpha, int32_t max_depth, const std::vector<int>& table,
              int depth0, int reps, float* ms, fbn_stats* st)
{
    fbn_handle* h = hs[0];
    apply_tuning(hs, k, table, depth0);
    int rc = run_skeleton(hs, k, alpha, max_depth);
    if (rc) return rc;
    cudaEvent_t e0 = h->ws.kev[0], e1 = h->ws.kev[1];
    std::vector<float> whole;
    std::vector<std::vector<double>> depth(FBN_MAX_DEPTHS);
    for (int r = 0; r < reps; ++r) {
        CK(cudaEventRecord(e0, h->stream));
        rc = run_skeleton(hs, k, alpha, max_depth);
        if (rc) return rc;
        CK(cudaEventRecord(e1, h->stream));
        CK(cudaEventSynchronize(e1));
        float t = 0.f;
        CK(cudaEventElapsedTime(&t, e0, e1));
        whole.push_back(t);
        for (int d = 0; d < FBN_MAX_DEPTHS; ++d) depth[d].push_back(h->stats.test_ms[d]);
    }
    auto median = [](auto v) {
        std::sort(v.begin(), v.end());
        return v[v.size() / 2];
    };
    *st = h->stats;
    *ms = median(whole);
    for (int d = 0; d < FBN_MAX_DEPTHS; ++d) st->test_ms[d] = median(depth[d]);
    return FBN_OK;
}

int autotune_impl(fbn_handle* const* hs, int k, double alpha, int32_t max_depth, fbn_tuning* out)
{
    fbn_handle* h = hs[0];
    const fbn_options& o = h->opt;
    const bool pool = o.form == FBN_FORM_POOL;
    // candidates for the pool depths: byte histograms at each group size, and
    // one-hot planes at the depths they serve (their pools run warp groups)
    std::vector<int> cands;
    if (pool && o.group_threads == 0) {
        for (int g : {32, 64, 128, kTestThreads}) cands.push_back(g | (o.count == FBN_COUNT_BITS ? 0 : kTuneNoBits));
        if (o.count == FBN_COUNT_AUTO) cands.push_back(0);
    } else {
        cands.push_back(0);
    }
    const bool gram_rule = pool && use_gram(hs, k, true);
    const bool tune_d0 = pool && o.depth0 == FBN_DEPTH0_AUTO && gram_rule;
    const int d0_rule = gram_rule ? FBN_DEPTH0_GRAM : FBN_DEPTH0_HIST;
    fbn_tuning rep{};
    std::vector<std::vector<double>> test_ms;
    fbn_stats st{};
    float ms = 0.f;
    int depths = 0;
    for (int c : cands) {
        std::vector<int> table(kMaxDepthRecords, c);
        const int rc = timed_run(hs, k, alpha, max_depth, table, d0_rule, 3, &ms, &st);
        if (rc) return rc;
        depths = st.depths;
        test_ms.emplace_back(st.test_ms, st.test_ms + FBN_MAX_DEPTHS);
        rep.candidates += 1;
    }
    // depth 0: the Gram against the histogram (the pool at later depths as the
    // first candidate), by the depth's device time
    int d0 = 0;
    if (tune_d0) {
        std::vector<int> table(kMaxDepthRecords, cands[0]);
        fbn_stats sg{}, sh{};
        int rc = timed_run(hs, k, alpha, max_depth, table, FBN_DEPTH0_GRAM, 3, &ms, &sg);
        if (!rc) rc = timed_run(hs, k, alpha, max_depth, table, FBN_DEPTH0_HIST, 3, &ms, &sh);
        if (rc) return rc;
        rep.candidates += 2;
        d0 = sh.ms[0] < sg.ms[0] ? FBN_DEPTH0_HIST : FBN_DEPTH0_GRAM;
    }
    // per depth the fastest candidate
    std::vector<int> best(kMaxDepthRecords, cands[0]);
    for (int d = 0; d < depths && d < FBN_MAX_DEPTHS; ++d) {
        size_t bi = 0;
        for (size_t i = 1; i < cands.size(); ++i)
            if (test_ms[i][d] < test_ms[bi][d]) bi = i;
        best[d] = cands[bi];
    }
    // the whole skeleton under the choices against the fixed rules; keep the faster
    fbn_stats s1{};
    float ms_fixed = 0.f, ms_tuned = 0.f;
    int rc = timed_run(hs, k, alpha, max_depth, {}, 0, 5, &ms_fixed, &s1);
    if (!rc) rc = timed_run(hs, k, alpha, max_depth, best, d0, 5, &ms_tuned, &s1);
    if (rc) return rc;
    rep.candidates += 2;
    TuneChoice choice;
    if (ms_tuned <= ms_fixed) {
        choice.table = best;
        choice.depth0 = d0;
    }
    const bool gram_used = choice.depth0 ? choice.depth0 == FBN_DEPTH0_GRAM : gram_rule;
    rep.depths = depths;
    rep.depth0 = gram_used ? FBN_DEPTH0_GRAM : FBN_DEPTH0_HIST;
    apply_tuning(hs, k, choice.table, choice.depth0);
    const DepthPlan plan = depth_plan(hs, k, false);
    for (int d = 0; d < depths && d < FBN_MAX_DEPTHS; ++d) {
        const int c = choice.table.empty() ? 0 : choice.table[d];
        const bool bits = d == 0 ? plan.popc0 : d == 1 && plan.marg1;
        rep.count[d] = bits ? FBN_COUNT_BITS : FBN_COUNT_HIST;
        rep.group_threads[d] = bits ? 32 : o.group_threads ? o.group_threads : (c & kTuneGroupMask);   // 0: cost model
    }
    rep.ms_fixed = ms_fixed;
    rep.ms_tuned = ms_tuned;
    choice.report = rep;
    {
        std::lock_guard<std::mutex> lock(g_tune_mu);
        g_tune_cache[tune_key(hs, k, alpha, max_depth)] = choice;
    }
    if (out) *out = rep;
    return FBN_OK;
}

// FBN_TUNE_AUTO: the first skeleton call on a shape takes the cached choices
// of this device and shape, or tunes.
int ensure_tuned(fbn_handle* const* hs, int k, double alpha, int32_t max_depth)
{
    fbn_handle* h = hs[0];
    if (h->opt.tune != FBN_TUNE_AUTO) return FBN_OK;
    const std::vector<long long> key = tune_key(hs, k, alpha, max_depth);
    {
        std::lock_guard<std::mutex> lock(g_tune_mu);
        auto it = g_tune_cache.find(key);
        if (it != g_tune_cache.end()) {
            apply_tuning(hs, k, it->second.table, it->second.depth0);
            return FBN_OK;
        }
    }
    return autotune_impl(hs, k, alpha, max_depth, nullptr);
}

void free_handle(fbn_handle* h)
{
    if (!h) return;
    cudaSetDevice(h->device);
    if (h->stream) cudaStreamSynchronize(h->stream);
    set_snapshot(h, nullptr);
    h->ws.release();
    dfree(h->d_data); dfree(h->d_planes); dfree(h->d_ar); dfree(h->d_adj); dfree(h->d_nbr); dfree(h->d_eid); dfree(h->d_npos); dfree(h->d_deg);
    dfree(h->d_sep_len); dfree(h->d_sep_off);
    dfree(h->d_sep_cnt);
    dfree(h->d_bad); dfree(h->d_status); dfree(h->d_table); dfree(h->d_gscratch);
    dfree(h->d_off);
    if (h->h_table) cudaFreeHost(h->h_table);
    if (h->h_ci_out) cudaFreeHost(h->h_ci_out);
    if (h->h_status) cudaFreeHost(h->h_status);
    if (h->own_stream) cudaStreamDestroy(h->own_stream);
    delete h;
}

}  // namespace

void fbn::fbn_internal_set_error(const char* msg)
{
    g_create_error = msg;
}

// ==========================================================================
extern "C" {

int fbn_create(const uint8_t* data, int32_t n_vars, int64_t n_samples, const uint8_t* arities,
               const fbn_options* opt, fbn_handle** out)
{
    fbn_handle* h = nullptr;
    if (!out) return fail(nullptr, FBN_EINVAL, "out is NULL");
    *out = nullptr;
    if (!data || !arities) return fail(nullptr, FBN_EINVAL, "data or arities is NULL");
    if (n_vars < 2 || n_vars > kMaxVars)
        return fail(nullptr, FBN_EINVAL, "n_vars=%d outside [2, %d]", n_vars, kMaxVars);
    if (n_samples < 1 || n_samples >= (1LL << 31)) return fail(nullptr, FBN_EINVAL, "n_samples=%lld outside [1, 2^31)", (long long)n_samples);
    fbn_options o{};
    o.device = -1;
    if (opt) {
        o = *opt;
        for (int k = 0; k < 4; ++k)
            if (o.reserved[k]) return fail(nullptr, FBN_EINVAL, "reserved option field %d is nonzero", k);
        if (o.loop != FBN_LOOP_DEVICE && o.loop != FBN_LOOP_HOST) return fail(nullptr, FBN_EINVAL, "bad loop %d", o.loop);
        if (o.wait_limit < -1) return fail(nullptr, FBN_EINVAL, "bad wait_limit %d", o.wait_limit);
        if (o.group_threads != 0 && o.group_threads != 32 && o.group_threads != 64 && o.group_threads != 128 &&
            o.group_threads != kTestThreads)
            return fail(nullptr, FBN_EINVAL, "bad group_threads %d", o.group_threads);
        if (o.form != FBN_FORM_POOL && o.form != FBN_FORM_PLAIN) return fail(nullptr, FBN_EINVAL, "bad form %d", o.form);
        if (o.group_size < 0) return fail(nullptr, FBN_EINVAL, "bad group_size %d", o.group_size);
        if (o.depth0 < FBN_DEPTH0_AUTO || o.depth0 > FBN_DEPTH0_GRAM) return fail(nullptr, FBN_EINVAL, "bad depth0 %d", o.depth0);
        if (o.depth1 < FBN_DEPTH1_AUTO || o.depth1 > FBN_DEPTH1_TENSOR) return fail(nullptr, FBN_EINVAL, "bad depth1 %d", o.depth1);
        if (o.statistic != FBN_STAT_G2 && o.statistic != FBN_STAT_X2)
            return fail(nullptr, FBN_EINVAL, "bad statistic %d", o.statistic);
        if (o.df_mode != FBN_DF_FIXED && o.df_mode != FBN_DF_ADJUSTED)
            return fail(nullptr, FBN_EINVAL, "bad df_mode %d", o.df_mode);
        if (o.count < FBN_COUNT_AUTO || o.count > FBN_COUNT_BITS) return fail(nullptr, FBN_EINVAL, "bad count %d", o.count);
        if (o.tune != FBN_TUNE_OFF && o.tune != FBN_TUNE_AUTO) return fail(nullptr, FBN_EINVAL, "bad tune %d", o.tune);
        if (o.depth1 == FBN_DEPTH1_TENSOR && (o.statistic != FBN_STAT_G2 || o.df_mode != FBN_DF_FIXED))
            return fail(nullptr, FBN_EINVAL, "depth1 tensor takes the G^2 statistic with fixed df only");
    }
    int max_ar = 0;
    for (int v = 0; v < n_vars; ++v) {
        if (arities[v] < 2) return fail(nullptr, FBN_EINVAL, "arity of variable %d is %d < 2", v, arities[v]);
        max_ar = std::max(max_ar, (int)arities[v]);
    }
    if (o.depth1 == FBN_DEPTH1_TENSOR && max_ar > nbr1_max_arity())
        return fail(nullptr, FBN_EINVAL, "depth1 tensor takes arities <= %d, not %d", nbr1_max_arity(), max_ar);
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) {
        cudaGetLastError();
        return fail(nullptr, FBN_ECUDA, "no CUDA device available");
    }
    int dev = o.device;
    if (dev < 0) {
        if (cudaGetDevice(&dev) != cudaSuccess) return fail(nullptr, FBN_ECUDA, "cudaGetDevice failed");
    }
    if (dev >= ndev) return fail(nullptr, FBN_EINVAL, "device %d of %d", dev, ndev);
    if (cudaSetDevice(dev) != cudaSuccess) return fail(nullptr, FBN_ECUDA, "cudaSetDevice(%d) failed", dev);

    h = new fbn_handle();
    h->device = dev;
    h->opt = o;
    h->n = n_vars;
    h->N = n_samples;
    h->ld = (n_samples + 255) / 256 * 256;
    h->max_arity = max_ar;
    h->h_ar.assign(arities, arities + n_vars);
    auto bail = [&](int code) {
        std::string m = h->err;
        free_handle(h);
        g_create_error = m;
        return code;
    };
#define CKC(call)                                                                          \
    do {                                                                                   \
        cudaError_t e_ = (call);                                                           \
        if (e_ != cudaSuccess) {                                                           \
            fail(h, e_ == cudaErrorMemoryAllocation ? FBN_ENOMEM : FBN_ECUDA, "%s: %s", #call, \
                 cudaGetErrorString(e_));                                                  \
            return bail(e_ == cudaErrorMemoryAllocation ? FBN_ENOMEM : FBN_ECUDA);           \
        }                                                                                  \
    } while (0)
    CKC(cudaStreamCreateWithFlags(&h->own_stream, cudaStreamNonBlocking));
    h->stream = h->own_stream;
    const size_t nn = (size_t)n_vars * n_vars;
    CKC(dalloc(&h->d_data, (size_t)n_vars * h->ld));
    h->plane_ld = ((n_samples + 31) / 32 + 3) / 4 * 4;   // 32-sample words, whole uint4 groups
    h->nplanes = max_ar <= kMargMaxArity ? max_ar - 1 : 0;
    CKC(dalloc(&h->d_planes, (size_t)n_vars * h->nplanes * h->plane_ld));
    CKC(dalloc(&h->d_ar, n_vars));
    CKC(dalloc(&h->d_adj, (nn + 15) / 16 * 16));   // read in whole 16-byte words
    CKC(dalloc(&h->d_nbr, nn));
    CKC(dalloc(&h->d_eid, nn));
    CKC(dalloc(&h->d_npos, nn));
    CKC(dalloc(&h->d_deg, n_vars));
    CKC(dalloc(&h->d_sep_len, nn));
    CKC(dalloc(&h->d_sep_off, nn));
    CKC(dalloc(&h->d_bad, 1));
    CKC(dalloc(&h->d_status, 1));
    CKC(cudaMallocHost((void**)&h->h_ci_out, 3 * sizeof(double)));
    CKC(cudaMallocHost((void**)&h->h_status, sizeof(unsigned long long)));
    CKC(cudaHostGetDevicePointer((void**)&h->ci_out_dev, h->h_ci_out, 0));
    CKC(cudaHostGetDevicePointer((void**)&h->status_dev, h->h_status, 0));
    cudaStream_t st = h->stream;
    CKC(cudaMemsetAsync(h->d_data, 0, (size_t)n_vars * h->ld, st));
    CKC(cudaMemsetAsync(h->d_eid, 0, nn * sizeof(int32_t), st));
    CKC(cudaMemsetAsync(h->d_bad, 0xff, sizeof(unsigned long long), st));
    CKC(cudaMemcpyAsync(h->d_ar, arities, n_vars, cudaMemcpyHostToDevice, st));
    std::vector<int32_t> off(2 * (size_t)n_vars);
    int M = 0;
    for (int v = 0; v < n_vars; ++v) {
        off[v] = M;
        off[n_vars + v] = M - v;
        M += arities[v];
    }
    h->M = M;
    h->Mp = gram_rows_padded(M);
    h->Mr = gram_rows_padded(M - n_vars);
    h->K = gram_samples_padded(n_samples);
    CKC(dalloc(&h->d_off, off.size()));
    CKC(cudaMemcpyAsync(h->d_off, off.data(), off.size() * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    // values must lie below their arity: checked on the device
    if (const int irc = ingest(h, data, h->d_bad, st)) return bail(irc);
    unsigned long long first_bad = 0;
    CKC(cudaMemcpyAsync(h->h_status, h->d_bad, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
    CKC(cudaStreamSynchronize(st));
    std::memcpy(&first_bad, h->h_status, sizeof first_bad);
    if (first_bad != ~0ULL) {
        const long long v = (long long)(first_bad / (unsigned long long)n_samples);
        const long long s = (long long)(first_bad % (unsigned long long)n_samples);
        fail(h, FBN_EDATA, "value of variable %lld at sample %lld is >= its arity %d", v, s, (int)arities[v]);
        return bail(FBN_EDATA);
    }
#undef CKC
    *out = h;
    return FBN_OK;
}

int fbn_update_data(fbn_handle* h, const uint8_t* data)
{
    if (!h) return FBN_EINVAL;
    if (!data) return fail(h, FBN_EINVAL, "data is NULL");
    CK(cudaSetDevice(h->device));
    cudaStream_t st = h->stream;
    h->learnt = false;
    drop_sepsets(h);
    const int prc = ingest(h, data, h->d_bad, st);
    if (prc) return prc;
    CK(cudaMemcpyAsync(h->h_status, h->d_bad, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    unsigned long long first_bad;
    std::memcpy(&first_bad, h->h_status, sizeof first_bad);
    if (first_bad != ~0ULL) {
        CK(cudaMemsetAsync(h->d_bad, 0xff, sizeof(unsigned long long), st));   // all ones between calls
        CK(cudaStreamSynchronize(st));                                         // whatever the next call's stream
        const long long v = (long long)(first_bad / (unsigned long long)h->N);
        const long long smp = (long long)(first_bad % (unsigned long long)h->N);
        return fail(h, FBN_EDATA, "value of variable %lld at sample %lld is >= its arity %d", v, smp,
                    (int)h->h_ar[v]);
    }
    return FBN_OK;
}

int fbn_update_data_batch(fbn_handle* const* hs, int32_t k, const uint8_t* const* data)
{
    if (!hs || k < 1 || !hs[0] || !data) return FBN_EINVAL;
    fbn_handle* h = hs[0];
    for (int p = 0; p < k; ++p) {
        if (!hs[p]) return fail(h, FBN_EINVAL, "handle %d is NULL", p);
        if (!data[p]) return fail(h, FBN_EINVAL, "data %d is NULL", p);
        if (hs[p]->device != h->device) return fail(h, FBN_EINVAL, "handle %d is on another device", p);
    }
    CK(cudaSetDevice(h->device));
    cudaStream_t st = h->stream;
    Workspace& ws = h->ws;
    if ((size_t)k > ws.bad_cap) {   // one flag per data set
        dfree(ws.d_bads);
        if (ws.h_bads) cudaFreeHost(ws.h_bads);
        ws.d_bads = ws.h_bads = nullptr;
        ws.bad_cap = 0;
        CK(dalloc(&ws.d_bads, k));
        CK(cudaMallocHost((void**)&ws.h_bads, k * sizeof(unsigned long long)));
        ws.bad_cap = (size_t)k;
    }
    CK(cudaMemsetAsync(ws.d_bads, 0xff, k * sizeof(unsigned long long), st));
    for (int p = 0; p < k; ++p) {   // every data set queued on one stream
        fbn_handle* q = hs[p];
        q->learnt = false;
        drop_sepsets(q);
        const int prc = ingest(q, data[p], ws.d_bads + p, st);
        if (prc) return fail(h, prc, "%s", q->err.c_str());
    }
    CK(cudaMemcpyAsync(ws.h_bads, ws.d_bads, k * sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    for (int p = 0; p < k; ++p) {
        const fbn_handle* q = hs[p];
        const unsigned long long first_bad = ws.h_bads[p];
        if (first_bad != ~0ULL) {
            const long long v = (long long)(first_bad / (unsigned long long)q->N);
            const long long smp = (long long)(first_bad % (unsigned long long)q->N);
            return fail(h, FBN_EDATA, "data set %d: value of variable %lld at sample %lld is >= its arity %d", p, v, smp,
                        (int)q->h_ar[v]);
        }
    }
    return FBN_OK;
}

int fbn_set_stream(fbn_handle* h, void* stream)
{
    if (!h) return FBN_EINVAL;
    h->stream = stream ? (cudaStream_t)stream : h->own_stream;
    return FBN_OK;
}

int fbn_ci_test(fbn_handle* h, int32_t x, int32_t y, const int32_t* z, int32_t nz, double* g2, double* df,
                double* p)
{
    if (!h) return FBN_EINVAL;
    if (!g2 || !df || !p) return fail(h, FBN_EINVAL, "null output pointer");
    long long cells = 0;
    int rc = check_test_args(h, x, y, z, nz, &cells);
    if (rc) return rc;
    rc = run_ci(h, x, y, z, nz, cells, false);
    if (rc) return rc;
    *g2 = h->h_ci_out[0];
    *df = h->h_ci_out[1];
    *p = h->h_ci_out[2];
    return FBN_OK;
}

int fbn_ci_table(fbn_handle* h, int32_t x, int32_t y, const int32_t* z, int32_t nz, int32_t* counts, int64_t cap)
{
    if (!h) return FBN_EINVAL;
    if (!counts) return fail(h, FBN_EINVAL, "counts is NULL");
    long long cells = 0;
    int rc = check_test_args(h, x, y, z, nz, &cells);
    if (rc) return rc;
    if (cap < cells) return fail(h, FBN_EINVAL, "cap %lld < %lld cells", (long long)cap, cells);
    rc = run_ci(h, x, y, z, nz, cells, true);
    if (rc) return rc;
    if (cells <= kCiHostTable) std::memcpy(counts, h->h_table, cells * sizeof(int32_t));
    else CK(cudaMemcpy(counts, h->d_table, cells * sizeof(int32_t), cudaMemcpyDeviceToHost));
    return FBN_OK;
}

int fbn_learn_skeleton(fbn_handle* h, double alpha, int32_t max_depth, uint8_t* adj_out)
{
    if (!h) return FBN_EINVAL;
    drop_sepsets(h);
    if (!(alpha > 0.0 && alpha < 1.0)) return fail(h, FBN_EINVAL, "alpha=%g outside (0, 1)", alpha);
    if (max_depth < -1) return fail(h, FBN_EINVAL, "max_depth=%d < -1", max_depth);
    h->learnt = false;
    fbn_handle* hs[1] = {h};
    uint8_t* outs[1] = {adj_out};
    const int rc = ensure_tuned(hs, 1, alpha, max_depth);
    if (rc) return rc;
    return run_skeleton(hs, 1, alpha, max_depth, outs);
}

int fbn_learn_skeleton_batch(fbn_handle* const* hs, int32_t k, double alpha, int32_t max_depth,
                             uint8_t* const* adj_out)
{
    if (!hs || k < 1) return FBN_EINVAL;
    fbn_handle* h = hs[0];
    for (int p = 0; p < k; ++p) {
        if (!hs[p]) return fail(h, FBN_EINVAL, "handle %d is NULL", p);
        if (hs[p]->device != h->device) return fail(h, FBN_EINVAL, "handle %d is on another device", p);
        hs[p]->learnt = false;
        drop_sepsets(hs[p]);
    }
    if (!(alpha > 0.0 && alpha < 1.0)) return fail(h, FBN_EINVAL, "alpha=%g outside (0, 1)", alpha);
    if (max_depth < -1) return fail(h, FBN_EINVAL, "max_depth=%d < -1", max_depth);
    const int rc = ensure_tuned(hs, k, alpha, max_depth);
    if (rc) return rc;
    return run_skeleton(hs, k, alpha, max_depth, adj_out);
}

int fbn_learn_skeleton_sharded(fbn_handle* h, double alpha, int32_t max_depth, fbn_shard_own_fn own,
                               fbn_shard_exchange_fn exchange, void* ctx, uint8_t* adj_out)
{
    if (!h) return FBN_EINVAL;
    drop_sepsets(h);
    h->learnt = false;
    if (!own || !exchange) return fail(h, FBN_EINVAL, "own and exchange callbacks are required");
    if (!(alpha > 0.0 && alpha < 1.0)) return fail(h, FBN_EINVAL, "alpha=%g outside (0, 1)", alpha);
    if (max_depth < -1) return fail(h, FBN_EINVAL, "max_depth=%d < -1", max_depth);
    fbn_handle* hs[1] = {h};
    uint8_t* outs[1] = {adj_out};
    const ShardHooks hooks{own, exchange, ctx};
    return run_skeleton(hs, 1, alpha, max_depth, outs, &hooks);
}

int fbn_autotune(fbn_handle* const* hs, int32_t k, double alpha, int32_t max_depth, fbn_tuning* out)
{
    if (!hs || k < 1 || !hs[0]) return FBN_EINVAL;
    fbn_handle* h = hs[0];
    for (int p = 0; p < k; ++p) {
        if (!hs[p]) return fail(h, FBN_EINVAL, "handle %d is NULL", p);
        if (hs[p]->device != h->device) return fail(h, FBN_EINVAL, "handle %d is on another device", p);
        hs[p]->learnt = false;
        drop_sepsets(hs[p]);
    }
    if (!(alpha > 0.0 && alpha < 1.0)) return fail(h, FBN_EINVAL, "alpha=%g outside (0, 1)", alpha);
    if (max_depth < -1) return fail(h, FBN_EINVAL, "max_depth=%d < -1", max_depth);
    return autotune_impl(hs, k, alpha, max_depth, out);
}

int fbn_pairwise_counts(fbn_handle* h, int32_t* counts, int64_t cap)
{
    if (!h) return FBN_EINVAL;
    if (!counts) return fail(h, FBN_EINVAL, "counts is NULL");
    const long long MM = (long long)h->M * h->M;
    if (cap < MM) return fail(h, FBN_EINVAL, "cap %lld < M*M = %lld", (long long)cap, MM);
    CK(cudaSetDevice(h->device));
    Workspace& ws = h->ws;
    fbn_handle* hs[1] = {h};
    int rc = grow_workspace(h, ws, (long long)h->n * (h->n - 1) / 2, h->n, 1, h->n);
    if (rc) return rc;
    ProblemDev P{};
    P.data = h->d_data; P.ar = h->d_ar; P.adj = h->d_adj; P.nbr = h->d_nbr; P.eid = h->d_eid; P.npos = h->d_npos; P.deg = h->d_deg;
    P.sep_len = h->d_sep_len; P.sep_off = h->d_sep_off; P.ld = h->ld; P.n = h->n; P.N = (int32_t)h->N;
    P.max_arity = h->max_arity;
    rc = prepare_gram(hs, 1, ws, &P);
    if (rc) return rc;
    // straight into a device buffer of the caller's; else through the workspace
    const bool device_out = ((uintptr_t)counts & 3) == 0 && device_range(counts, (size_t)MM * sizeof(int32_t), h->device, false);
    if (!device_out) {
        rc = prepare_pairs(hs, 1, ws, &P);
        if (rc) return rc;
    }
    std::vector<int32_t> vp(h->n, 0), vf(1, 0);
    ws.up_last.clear();   // the skeleton's next call uploads its own descriptors again
    CK(cudaMemcpyAsync(ws.probs, &P, sizeof P, cudaMemcpyHostToDevice, h->stream));
    CK(cudaMemcpyAsync(ws.vtx_prob, vp.data(), h->n * sizeof(int32_t), cudaMemcpyHostToDevice, h->stream));
    CK(cudaMemcpyAsync(ws.vtx_first, vf.data(), sizeof(int32_t), cudaMemcpyHostToDevice, h->stream));
    CK(cudaMemsetAsync(h->d_status, 0, sizeof(unsigned), h->stream));
    rc = run_gram(h, ws, 1, h->n, h->d_status);
    if (rc) return rc;
    PairsGramArgs pa;
    pa.emit = pa.sym = 1;
    pa.out = device_out ? counts : ws.gram_G;
    pa.ldo = h->M;
    pa.max_arity = h->max_arity;
    int sms = 0;
    CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device));
    CK(launch_pairs_gram(ws.probs, ws.vtx_prob, ws.vtx_first, h->n, h->n, pa, sms, h->stream));
    if (!device_out)
        CK(cudaMemcpyAsync(counts, ws.gram_G, (size_t)MM * sizeof(int32_t), cudaMemcpyDefault, h->stream));
    CK(cudaMemcpyAsync(h->h_status, h->d_status, sizeof(unsigned), cudaMemcpyDeviceToHost, h->stream));
    CK(cudaStreamSynchronize(h->stream));
    return check_status(h, *h->h_status);
}

int32_t fbn_get_sepset(const fbn_handle* hc, int32_t i, int32_t j, int32_t* buf, int32_t cap)
{
    if (!hc || !hc->learnt) return FBN_EINVAL;
    fbn_handle* h = const_cast<fbn_handle*>(hc);   // the host copy is a cache of device results
    if (h->sep_pending) {
        const int rc = materialize_sepsets(h, h->ws);
        if (rc) return rc;
    }
    if (i < 0 || j < 0 || i >= h->n || j >= h->n || i == j) return FBN_EINVAL;
    if (i > j) std::swap(i, j);
    const long long k = find_sepset(h, i, j);
    if (k < 0) return -1;
    const int32_t L = (int32_t)(csr_end(h, k) - h->csr_offs[k]);
    if (L > 0 && cap > 0 && !buf) return FBN_EINVAL;
    for (int t = 0; t < L && t < cap; ++t) buf[t] = h->csr_members[(size_t)h->csr_offs[k] + t];
    return L;
}

int fbn_export_sepsets(const fbn_handle* hc, int64_t* n_removed, int64_t* n_members, int32_t* pairs,
                       int64_t* offsets, int32_t* members)
{
    if (!hc || !hc->learnt || !n_removed || !n_members) return FBN_EINVAL;
    fbn_handle* h = const_cast<fbn_handle*>(hc);   // the host copy is a cache of device results
    if (h->sep_pending) {
        const int rc = materialize_sepsets(h, h->ws);
        if (rc) return rc;
    }
    const int64_t nr = h->csr_R, nm = h->csr_M;
    if (pairs && nr > 0) std::memcpy(pairs, h->csr_pairs, 2 * (size_t)nr * sizeof(int32_t));
    if (offsets && nr > 0) std::memcpy(offsets, h->csr_offs, (size_t)nr * sizeof(int64_t));
    if (members && nm > 0) std::memcpy(members, h->csr_members, (size_t)nm * sizeof(int32_t));
    if (offsets) offsets[nr] = nm;
    *n_removed = nr;
    *n_members = nm;
    return FBN_OK;
}

int fbn_orient_cpdag(const fbn_handle* hc, uint8_t* cpdag_out)
{
    if (!hc || !hc->learnt || !cpdag_out) return FBN_EINVAL;
    fbn_handle* h = const_cast<fbn_handle*>(hc);   // the host copy is a cache of device results
    if (h->sep_pending) {
        const int rc = materialize_sepsets(h, h->ws);
        if (rc) return rc;
    }
    const int n = h->n;
    const size_t nn = (size_t)n * n;
    std::vector<uint8_t> A(nn);
    CK(cudaSetDevice(h->device));
    CK(cudaMemcpyAsync(A.data(), h->d_adj, nn, cudaMemcpyDeviceToHost, h->stream));
    CK(cudaStreamSynchronize(h->stream));
    std::vector<std::vector<int>> nb(n);
    for (int u = 0; u < n; ++u)
        for (int v = 0; v < n; ++v)
            if (A[(size_t)u * n + v]) nb[u].push_back(v);
    auto adj = [&](int u, int v) { return A[(size_t)u * n + v] != 0; };
    auto in_sepset = [&](int a, int b, int k) {   // a < b, not adjacent
        const long long r = find_sepset(h, a, b);
        if (r < 0) return false;
        for (int64_t t = h->csr_offs[r]; t < csr_end(h, r); ++t)
            if (h->csr_members[(size_t)t] == k) return true;
        return false;
    };
    // step 2: arrowheads of the unshielded colliders
    std::vector<uint8_t> head(nn, 0);   // head[a*n+k]: a -> k marked
    for (int k = 0; k < n; ++k) {
        const std::vector<int>& N = nb[k];
        for (size_t x = 0; x < N.size(); ++x)
            for (size_t y = x + 1; y < N.size(); ++y) {
                const int a = N[x], b = N[y];
                if (adj(a, b) || in_sepset(a, b, k)) continue;
                head[(size_t)a * n + k] = 1;
                head[(size_t)b * n + k] = 1;
            }
    }
    std::vector<uint8_t> arc(nn, 0);    // arc[a*n+b]: a -> b oriented
    for (size_t e = 0; e < nn; ++e) {
        const size_t a = e / n, b = e % n;
        if (head[e] && !head[b * n + a]) arc[e] = 1;
    }
    auto open = [&](int u, int v) { return adj(u, v) && !arc[(size_t)u * n + v] && !arc[(size_t)v * n + u]; };
    // step 3: Meek rules in rounds
    std::vector<std::pair<int, int>> found;
    std::vector<uint8_t> want(nn, 0);
    for (;;) {
        found.clear();
        for (int b = 0; b < n; ++b)
            for (int c : nb[b]) {
                if (!open(b, c)) continue;
                bool orient = false;
                for (int a : nb[b]) {
                    if (a != c && arc[(size_t)a * n + b] && !adj(a, c)) orient = true;      // R1
                    if (arc[(size_t)b * n + a] && arc[(size_t)a * n + c]) orient = true;  // R2
                    if (orient) break;
                }
                if (!orient) {   // R3: two non-adjacent m1, m2 with b - m -> c
                    std::vector<int> mids;
                    for (int m : nb[b])
                        if (open(b, m) && arc[(size_t)m * n + c]) mids.push_back(m);
                    for (size_t x = 0; x < mids.size() && !orient; ++x)
                        for (size_t y = x + 1; y < mids.size(); ++y)
                            if (!adj(mids[x], mids[y])) {
                                orient = true;
                                break;
                            }
                }
                if (orient) {
                    found.emplace_back(b, c);
                    want[(size_t)b * n + c] = 1;
                }
            }
        bool changed = false;
        for (const auto& bc : found) {
            const size_t fw = (size_t)bc.first * n + bc.second, bw = (size_t)bc.second * n + bc.first;
            if (!want[bw]) {
                arc[fw] = 1;
                changed = true;
            }
        }
        for (const auto& bc : found) want[(size_t)bc.first * n + bc.second] = 0;
        if (!changed) break;
    }
    for (size_t e = 0; e < nn; ++e) {
        const size_t a = e / n, b = e % n;
        cpdag_out[e] = (A[e] && !arc[b * n + a]) ? 1 : 0;
    }
    return FBN_OK;
}

int fbn_get_stats(const fbn_handle* h, fbn_stats* out)
{
    if (!h || !out) return FBN_EINVAL;
    *out = h->stats;
    return FBN_OK;
}

const char* fbn_last_error(const fbn_handle* h)
{
    return h ? h->err.c_str() : g_create_error.c_str();
}

void fbn_destroy(fbn_handle* h)
{
    free_handle(h);
}

}  // extern "C"
