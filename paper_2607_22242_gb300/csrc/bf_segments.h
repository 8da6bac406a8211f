// bf_segments.h -- internal interface between the C ABI and the kernels of
// scenarios cut by barriers (bf_segments.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "bf_launch.h"
#include "bf_segments.cuh"
#include "bf_tree.h"

namespace bfk {

// State of one launch of the optimum kernel in device memory: each table's
// best key so far, and the blocks that have finished.  It holds (~0, ..., 0)
// between launches.
struct SegSync {
  unsigned long long key[kSegMax / 2];
  uint32_t blocks_done;
  uint32_t pad;
};

// Simulate the segments of two or more tools into table[plan.entries].
cudaError_t launch_segment_tables(const SegPlan& plan, uint32_t* table, cudaStream_t st);

// Every makespan and feasibility flag of the sums' mappings; launched right
// after launch_segment_tables on the same stream.
cudaError_t launch_segment_eval(const SegSums& sums, const uint32_t* table, uint32_t* ms, uint8_t* fe, cudaStream_t st);

// The optimum (makespan, lowest canonical index) of the full (radix 3) or the
// binary cpu/gpu_now space (radix 2) to *host_best, pinned host memory as the
// device addresses it.
cudaError_t launch_segment_optimum(const SegPlan& plan, uint32_t radix, SegSync* sync, BestRecord* host_best,
                                   cudaStream_t st);

}  // namespace bfk
