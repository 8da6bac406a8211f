// bf_tree.h -- internal interface between the C ABI (bf_capi.cu) and the tree
// search kernels (bf_tree.cu): the best-so-far record, the counters and the
// launchers.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "bf_tree.cuh"

namespace bfk {

// Best mapping found so far: makespan, then canonical index (lexicographic
// minimum, updated by 16-byte compare-and-swap).  {~0, ~0} = none.
struct __align__(16) BestRecord {
  unsigned long long ms;
  unsigned long long idx;
};

// Device-side counters of one tree search.
struct TreeCounters {
  unsigned long long nodes;       // nodes appended to any level
  unsigned long long leaf_nodes;  // leaf-level nodes enumerated (counted by the warp task of their first chunk)
  unsigned long long leaves;      // mappings simulated by the leaf kernel
  uint32_t incumbent;             // the starting bound
  uint32_t error;                 // bit 0: a level buffer overflowed; bit 1: a best-record update gave up
};

// A level of the search: its node buffer, and how many nodes have been
// appended to it since it was last emptied (in device memory).
struct TreeLevel {
  uint32_t* buf;
  uint32_t* count;
};

size_t tree_node_words();
// The starting bound: the least feasible of n candidates' makespans
// (0xFFFFFFFF without one), to bounds->live and ctr->incumbent.
cudaError_t launch_tree_bound(const uint32_t* ms, const uint8_t* fe, uint32_t n, TreeBounds* bounds, TreeCounters* ctr,
                              cudaStream_t st);
// Append the surviving nodes of the first d0 tools' modes to `dst` (level d0).
cudaError_t launch_tree_start(const TablesW& tb, const TreeConsts& tc, uint32_t d0, TreeLevel dst, uint32_t cap,
                              TreeBounds* bounds, TreeCounters* ctr, cudaStream_t st);
// Expand the last min(*src.count, pop) nodes of `src` (level d, at most
// most_nodes of them) into `dst`; the counts are read on the device, so that
// launches follow one another without the host.
cudaError_t launch_tree_expand(const TablesW& tb, const TreeConsts& tc, TreeLevel src, uint32_t pop,
                               uint32_t most_nodes, uint32_t d, TreeLevel dst, uint32_t cap, TreeBounds* bounds,
                               TreeCounters* ctr, cudaStream_t st);
// Enumerate the leaves of every node of `src`, the leaf level.  A start or an
// expansion must have run since the last launch of this (TreeBounds::leaf).
cudaError_t launch_tree_leaf(const TablesW& tb, const TreeConsts& tc, TreeLevel src, uint32_t cap,
                             uint32_t most_nodes, TreeBounds* bounds, BestRecord* best, TreeCounters* ctr,
                             cudaStream_t st);

}  // namespace bfk
