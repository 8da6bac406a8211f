// bf_capi_internal.h -- what the C ABI's translation units share: the
// handle and its scratch, and the helpers for errors, allocation, bounded
// waits and index lists (defined in bf_capi.cu).  Not installed; not part of
// the ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/bf.h"
#include "bf_lanetree_launch.h"
#include "bf_launch.h"
#include "bf_plan.h"
#include "bf_scratch_pool.h"
#include "bf_segments.h"
#include "bf_tree.h"

// Per-handle scratch, one block on the device and a pinned mirror on the host:
// the launch states, the packed search key, the tree search's best record,
// bound and counters, and the what-if probe list with its results.
struct bf_scratch {
  // Set at creation: what searches expect to find (and leave) in device memory.
  struct Launch {
    bfk::SearchSync search;  // whole-space searches; search.key of the host mirror receives their result
    bfk::SegSync seg;        // branch and bound of scenarios cut by barriers
    bfk::LaneTreeRecord lt;  // whole-space search by the lane-tree kernel (bf_scenario::lanetree)
  } launch;
  unsigned long long key;
  uint32_t survivors;   // pruned search: number of surviving prefixes
  uint32_t pruned_bound;  // pruned search: the incumbent's makespan (set with survivors)
  bfk::BestRecord best;      // tree search: best (makespan, index) so far
  bfk::TreeBounds bounds;    // tree search: makespan bounds for pruning
  bfk::TreeCounters ctr;     // tree search: counters and error bits
  uint32_t count[BF_MAX_TOOLS + 1];  // tree search: nodes of each level
  uint64_t idx[BF_MAX_PROBES];
  uint32_t ms[BF_MAX_PROBES];
  uint8_t fe[BF_MAX_PROBES];
};

struct bf_scenario {
  bf_scenario_desc desc;
  bfk::TablesW wide;    // all n tools, 32 slots (index lists and the tree search)
  bfk::Tables tables;   // all n tools (n <= BF_MAX_TOOLS_ENUM; zero otherwise)
  bfk::Tables window;   // tools [W0, n), renumbered from 0
  bfk::Plan plan;       // enumeration split and window (see bfk::Plan), full range
  // Searches of the whole space: the tools renumbered with the sources first
  // (bf_plan.h relabel_sources_first; equal to the above when that order is
  // the scenario's own), with their split and window.
  bfk::Tables rtables;
  bfk::Tables rwindow;
  bfk::Plan rplan;
  bfk::Tables pwindow;  // bf_search_pruned: its window (of pplan, on rtables)
  bfk::Plan pplan;      // bf_search_pruned: its split (shorter prefixes: fewer to filter)
  // Searches of the whole space by the lane-tree kernel (scenarios of
  // kLtSingleMinTools to kLtMaxTools tools): its record's level boundary x
  // and the blocks of a launch; lanetree false otherwise.
  bool lanetree;
  uint32_t lt_x, lt_blocks;
  // Scenarios cut by barriers: the segments (seg.count = 0 otherwise), and
  // their tables, allocated by the first evaluation that uses them.
  bfk::SegPlan seg;
  uint32_t* d_table;
  int device;
  unsigned long long ctx;     // ID of the context the scratch was made in, 0 when it could not be told
  bf_scratch* d_scratch;      // device scratch
  bf_scratch* h_scratch;      // pinned host mirror
  unsigned long long* d_key;  // &d_scratch->key
  unsigned long long* h_key;  // &h_scratch->key
  bf_scratch* d_host_scratch; // h_scratch as the device addresses it
  uint32_t* d_survivors;      // pruned search: 3^pplan.P prefix slots, allocated on first use
  uint32_t* d_levels;         // tree search: node buffers of every level, allocated on first use
  size_t levels_bytes;
  bfcapi::OpenCalls calls;    // whose work may be in flight (also after one that failed or timed out)
};

namespace bfcapi {

// Record `code` and a printf-style message as this thread's last error; returns code.
int fail(int code, const char* fmt, ...);
// A failed CUDA call: BF_ENOMEM for allocation failures, else BF_ECUDA.
int cuda_fail(cudaError_t e, const char* what);
// cudaMalloc / cudaMallocHost with the test-only failure injection.
cudaError_t lib_malloc(void** p, size_t bytes);
cudaError_t lib_malloc_host(void** p, size_t bytes);
// Wait for `st` with the process-wide time limit (BF_ETIMEOUT when it passes).
int wait_stream(cudaStream_t st, const char* who);
// Around a handle's call that uses its scratch: work goes out; its last wait,
// after which (on BF_OK) nothing is in flight.
void begin_call(const bf_scenario* scn);
int end_call(const bf_scenario* scn, cudaStream_t st, const char* who);
// That limit in milliseconds (0: none).
uint32_t wait_limit_ms();
// BF_EINVAL unless the handle's device is current.
int check_device(const bf_scenario* scn, const char* who);
// The optimum of the full (radix 3) or binary space of a scenario cut by
// barriers (scn->seg.count != 0), by one launch and one bounded wait.
int segment_optimum(const bf_scenario* scn, uint32_t radix, bf_result* out, cudaStream_t st, const char* who);
// A best record as a search's result.
void fill_best(const volatile bfk::BestRecord& best, uint32_t n, bf_result* out);
// Makespans of a list of mappings on the index-list kernel.
cudaError_t launch_list(const bf_scenario* scn, const uint64_t* idx, uint64_t count, uint32_t* ms, uint8_t* fe,
                        cudaStream_t st);

}  // namespace bfcapi
