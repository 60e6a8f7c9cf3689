// Cluster flow solve: one system on one thread-block cluster, rows in level
// order, solutions passed between the cluster's SMs through distributed
// shared memory (flow.cu).
#pragma once

#include "solve.cuh"

namespace spt {

// Up to 32 rows of one level and one length class, 1 << llpr lanes per row:
// positions [base, base + cnt) of the flow order (level by level; inside a
// level by length class, then by row).
struct FlowGroup {
    int32_t base, cnt, llpr;
};

// What one lane of a group needs to know before its values come.
struct FlowLane {
    int32_t row;    // -1: no row
    uint32_t code;  // of the row's own position, see flow.cu
    uint32_t meta;  // blocks that depend on the row (16 bits), llpr (4), entries of the busiest lane (4)
    int32_t epoch;
};

// Schedule of one direction.  Slot g * 32 + l belongs to lane l of group g;
// the groups are sorted by block of the cluster.  A slot takes 60 bytes (FP64
// 80) and an entry 4 more; a row of up to 4 entries has one slot, of up to 16
// four, of up to 64 sixteen, a longer one 32, and the last group of a level and
// class is filled up to 32 slots.
struct FlowSched {
    const FlowLane *lanes;
    const uint4 *codes;    // of the lane's first four entries
    const int2 *src;       // position of the lane's first entry, and of the row's end (diagonal, forward)
    const uint32_t *ecode; // of every entry (read for the longest rows only)
    const int32_t *gptr;   // csize + 1: groups of every block
    void *vals;            // values of the lane's first four entries, refreshed by every solve
    void *inv;             // reciprocal diagonals, refreshed by every solve
    int32_t n, csize, ngroups;
};

constexpr int kFlowClasses = 4;
constexpr int kFlowMaxCluster = 16;
constexpr int64_t kFlowMaxRows = 900 * 1000 * 1000;  // generations of a slot fit 16 bits

// Plan-time tables of one direction; ptr/idx: CSR row pointers and columns
// (forward) or CSC column pointers and rows (transpose), lev: levels, L their
// number.  order, iperm: n entries (row at every position and its inverse);
// counts: L * kFlowClasses (rows per level and class); meta, mask: n entries
// of scratch.
cudaError_t flow_order(const int32_t *ptr, const int32_t *lev, int32_t n, int32_t L, bool trans, int32_t *order,
                       int32_t *iperm, int32_t *counts, cudaStream_t s, const Scratch *from);
cudaError_t flow_tables(const int32_t *ptr, const int32_t *idx, int32_t n, bool trans, bool f64, const int32_t *order,
                        const int32_t *iperm, const FlowGroup *groups, const int32_t *gptr, int32_t ngroups,
                        int32_t csize, uint32_t *meta, uint32_t *mask, FlowLane *lanes, uint4 *codes, int2 *src,
                        uint32_t *ecode, cudaStream_t s);

// Whether a cluster of `csize` blocks of the flow kernel can be resident.
bool flow_cluster_fits(int csize, bool f64);

template <class T>
cudaError_t solve_flow(const Sys<T> &A, const FlowSched &F, const Rhs<T> &R, bool trans, int32_t withhold,
                       const Waiter &w, cudaStream_t s);

}  // namespace spt
