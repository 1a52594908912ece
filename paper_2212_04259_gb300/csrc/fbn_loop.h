// fbn_loop.h -- the persistent depth loop of small problems (fbn_loop.cu).
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "fbn_internal.cuh"

namespace fbn {

constexpr int kTurnVertices = 128;   // variables of a problem whose depths one CTA prepares (fbn_turn.cuh)
constexpr int kTurnItems = 32768;    // items of a class it lays out
constexpr unsigned kLoopGaveUp = 1;      // a phase's wait ran out: the call starts over without the loop
constexpr unsigned kLoopHandedOver = 2;  // + d: the kernels of a depth go on at depth d ...
constexpr unsigned kLoopSplit = 1u << 16;   // ... and tests split by samples may not have run to their end

// Everything the loop's phases take, by value.
struct LoopArgs {
    const ProblemDev* probs;
    const int32_t *vtx_prob, *vtx_first;
    int total_vertices, max_n;
    int gs_forced;
    long long gs_edges;
    const long long* binom;
    int brows;
    long long warp_cells_cap;
    EdgeWork* edges;
    unsigned long long* min_accept;
    long long edge_cap;
    DepthCounters* ctr;
    unsigned long long *hist, *cursor;   // both classes, ord_cap entries each
    long long ord_cap;
    ScanClass sc[2];
    int32_t* sorted;
    double mean_n;
    int forced_group;
    long long split_stride;
    int need_marg;
    int32_t* sep_pool;
    long long sep_cap;
    DepthRecord* rec;
    int max_depth;
    int popc0, marg1;                    // depths 0 and 1 from one-hot planes
    PoolArgs small, big;                 // the two classes
    unsigned spin_limit;                 // polls of a phase barrier without progress before the loop gives up
    unsigned* left;                      // pinned host memory: how the loop ended early (below), 0 if it did not
    unsigned* bits;                      // one problem of <= kTurnVertices variables: its adjacency as a bit
                                         // matrix [kTurnVertices][kTurnVertices / 32] (nullptr: general phases only)
    unsigned* bar;                       // [2] arrivals of the current phase (and kGaveUp), phases opened so far
    DepthCounters init;                  // the counters' first state
    // one problem: results straight to pinned host memory (nullptr: left on
    // the device): counters, records, adjacency, and the separating sets as
    // CSR (removed pairs ascending, member offsets, members) with their totals
    DepthCounters* h_ctr;
    DepthRecord* h_rec;
    uint8_t* h_adj;
    int32_t* h_pairs;
    int64_t* h_offs;
    int32_t* h_members;
    long long* h_tot;
    long long* sep_cnt;                  // [2 n] row counts of the CSR (device)
};

cudaError_t prepare_loop(size_t smem_bytes, int* blocks_per_sm);
cudaError_t launch_loop(const LoopArgs& a, int grid, size_t smem_bytes, cudaStream_t st);

}  // namespace fbn
