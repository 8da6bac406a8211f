// bf_segments.cu -- kernels for scenarios cut by barriers (bf_segments.cuh):
//
//   segment_table_kernel  : simulates every mapping of every segment of two or
//                           more tools into its table (the lane tree of
//                           bf_lanetree.cuh with stores instead of a minimum).
//   segment_optimum_kernel: keeps each segment's best instead; its last block
//                           adds them up.
//   segment_eval_kernel   : sums over tiles of low parts times rows of high
//                           parts: every mapping of the range is one addition
//                           and one 5-byte store.
//   segment_direct_kernel : the same for scenarios with fewer low parts than a
//                           tile: both parts' sums in shared memory.
//
// The sums are launched as programmatic dependents of the tables, so their
// blocks start while the tables' last blocks run.
#include <cuda_runtime.h>

#include "bf_enum.cuh"
#include "bf_segments.h"

namespace bfk {
namespace {

using host::kSegDirect;
using host::kSegMaxRows;
using host::kSegPerThread;
using host::kSegThreads;
using host::kSegTile;

// Set a block up for its share of table t's roots: the record, its tables and
// the roots [3^x * j / blocks, 3^x * (j + 1) / blocks) of its place j among
// the table's blocks (radix^x roots for an optimum over two modes).
template <uint32_t NC>
__device__ __forceinline__ void seg_begin(const SegPlan& plan, uint32_t t, uint32_t x, uint32_t y, uint32_t radix,
                                          LtSharedT<NC>& S) {
  const uint32_t seg = plan.seg[t], lo = plan.start[seg], n = plan.start[seg + 1u] - lo;
  if (threadIdx.x < n) {
    const uint32_t v = threadIdx.x;
    S.rec.pred[v] = plan.pred[lo + v];
    for (uint32_t a = 0; a < 3; ++a) S.rec.dur[a][v] = plan.dur[a][lo + v];
    S.rec.vram[v] = plan.vram[lo + v];
    S.rec.pv[v] = plan.pv[lo + v];
  }
  if (threadIdx.x <= n) {
    S.rec.f[threadIdx.x] = plan.f[threadIdx.x];
    S.rec.frecip[threadIdx.x] = plan.frecip[threadIdx.x];
  }
  if (threadIdx.x == 0) {
    S.rec.n = n;
    S.rec.budget = plan.budget;
    S.rec.all_mask = (1u << n) - 1u;
    S.rec.x = x;
    S.rec.y = y;
    uint32_t roots = 1u, big = 0u;
    for (uint32_t v = 0; v < x; ++v) roots *= radix;
    for (uint32_t v = 0; v < n; ++v) big |= plan.vram[lo + v] > plan.budget ? 1u << v : 0u;
    S.rec.big_mask = big;
    const uint64_t j = blockIdx.x - plan.first_block[t], nb = plan.first_block[t + 1u] - plan.first_block[t];
    S.root_next = (uint32_t)(roots * j / nb);
    S.root_end = (uint32_t)(roots * (j + 1u) / nb);
  }
  __syncthreads();
  lt_fill_tables(S);
  __syncthreads();
}

// The table whose blocks include this one.
__device__ __forceinline__ uint32_t seg_table_of_block(const SegPlan& plan) {
  uint32_t t = 0u;
  while (t + 1u < plan.tables && plan.first_block[t + 1u] <= blockIdx.x) ++t;
  return t;
}

struct StoreTable {
  uint32_t* table;
  __device__ __forceinline__ void operator()(uint32_t idx, uint32_t ms) { table[idx] = ms; }
  __device__ __forceinline__ void dead(uint32_t idx) { table[idx] = kSegInfeasible; }
};

// Bound by the latency of a lane's simulation: one root per lane of a few
// blocks (7-tool segments of the 19-tool spine: 18 blocks, 11 us).
template <uint32_t NC>
__global__ void __launch_bounds__(kSegThreads, 5) segment_table_kernel(const __grid_constant__ SegPlan plan,
                                                                       uint32_t* table) {
  extern __shared__ uint32_t lt_rows_smem[];
  __shared__ LtSharedT<NC> S;
  cudaTriggerProgrammaticLaunchCompletion();
  const uint32_t t = seg_table_of_block(plan);
  seg_begin(plan, t, plan.x[t], plan.y[t], 3u, S);
  StoreTable sink{table + plan.off[plan.seg[t]]};
  LtSharedT<NC>& Sref = S;
  lt_lane<NC, false, true>(S, lt_rows_smem + threadIdx.x, blockDim.x,
                           [&Sref]() {
                             const uint32_t root = atomicAdd(&Sref.root_next, 1u);
                             return root < Sref.root_end ? root : 0xFFFFFFFFu;
                           },
                           sink);
}

// The optimum of the space of `radix` modes per tool (2: cpu and gpu_now, each
// tool a root digit, so that only such mappings are simulated).  Every block
// folds its best (makespan << 32 | segment mapping) into its segment's key;
// the last one adds the segments' bests up, hands the result to the host and
// leaves the launch state (~0, ..., 0) as the next launch expects it.
template <uint32_t NC>
__global__ void __launch_bounds__(kSegThreads, 5) segment_optimum_kernel(const __grid_constant__ SegPlan plan,
                                                                         uint32_t radix, SegSync* sync,
                                                                         BestRecord* host_best) {
  extern __shared__ uint32_t lt_rows_smem[];
  __shared__ LtSharedT<NC> S;
  if (plan.tables) {
    const uint32_t t = seg_table_of_block(plan), seg = plan.seg[t], n = plan.start[seg + 1u] - plan.start[seg];
    seg_begin(plan, t, radix == 2u ? n : plan.x[t], radix == 2u ? n : plan.y[t], radix, S);
    MinKeySink sink;
    LtSharedT<NC>& Sref = S;
    lt_lane<NC, false>(S, lt_rows_smem + threadIdx.x, blockDim.x,
                       [&Sref, radix]() {
                         const uint32_t root = atomicAdd(&Sref.root_next, 1u);
                         if (root >= Sref.root_end) return 0xFFFFFFFFu;
                         if (radix == 3u) return root;
                         uint32_t r = 0u, p = 1u;  // binary digits as base-3 digits
                         for (uint32_t m = root; m; m >>= 1, p *= 3u) r += (m & 1u) * p;
                         return r;
                       },
                       sink);
    unsigned long long best = sink.best;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = min(best, __shfl_xor_sync(0xFFFFFFFFu, best, o));
    if ((threadIdx.x & 31u) == 0u && best != ~0ull) atomicMin(&sync->key[t], best);
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  __threadfence();
  if (atomicAdd(&sync->blocks_done, 1u) != gridDim.x - 1u) return;
  unsigned long long ms = 0ull, idx = 0ull, place = 1ull;
  for (uint32_t j = 0, t = 0; j < plan.count; ++j) {
    uint32_t least = plan.alone[j][0], m = 0u;
    if (plan.size[j] == 3u) {
      for (uint32_t a = 1; a < radix; ++a)
        if (plan.alone[j][a] < least) {
          least = plan.alone[j][a];
          m = a;
        }
    } else {  // tables are in the segments' order; every segment has a feasible mapping (all cpu)
      const unsigned long long key = atomicExch(&sync->key[t++], ~0ull);
      least = (uint32_t)(key >> 32);
      m = (uint32_t)key;
    }
    ms += least;
    idx += m * place;
    place *= plan.size[j];
  }
  sync->blocks_done = 0u;
  host_best->ms = ms;
  host_best->idx = idx;
  __threadfence_system();
}

// The makespan written for a sum.
__device__ __forceinline__ uint32_t seg_makespan(uint32_t sum) { return sum < kSegInfeasible ? sum : kInfeasible; }

// The rows [h0, h1) of a block, and its low parts' sums.
struct SegTile {
  uint32_t x0, h0, h1;
  __device__ __forceinline__ explicit SegTile(const SegSums& s)
      : x0(blockIdx.x % s.x_tiles * kSegTile),
        h0(s.h_lo + blockIdx.x / s.x_tiles * s.rows),
        h1(min(h0 + s.rows, s.h_hi + 1u)) {}
};

// Thread t's low parts are x0 + t + 256 k.
__device__ __forceinline__ void seg_low_parts(const SegSums& s, const uint32_t* table, const SegTile& tile,
                                              uint32_t (&low)[kSegPerThread]) {
  uint32_t v[kSegPerThread];
#pragma unroll
  for (uint32_t k = 0; k < kSegPerThread; ++k) v[k] = min(tile.x0 + threadIdx.x + k * kSegThreads, s.A - 1u);
  segment_sum<kSegPerThread>(s, table, 0u, s.split, v, low);
}

// Tiled evaluation.  Each row of a block is kSegTile consecutive outputs (less
// at the edges), at any alignment; the low parts lie in shared memory in four
// interleaved planes (x mod 4), so that a thread reads the four that make one
// aligned 16-byte store of makespans and 4-byte store of flags without bank
// conflicts whatever the row's phase.  `aligned`: both output arrays have the
// same phase modulo 4 elements; else mapping by mapping.  Bound by the stores:
// 2^25 mappings, 168 MB, in 37 us (element-wise stores took 47,
// a row per block instead of per warp 41 with 60 % more instructions).
__global__ void __launch_bounds__(kSegThreads) segment_eval_kernel(const __grid_constant__ SegSums s,
                                                                   const uint32_t* table, uint32_t* ms, uint8_t* fe) {
  __shared__ uint32_t plane[4][kSegTile / 4], high[kSegMaxRows];
  cudaGridDependencySynchronize();
  const SegTile tile(s);
  for (uint32_t i = threadIdx.x; i < tile.h1 - tile.h0; i += kSegThreads)
    high[i] = segment_sum(s, table, s.split, s.count, tile.h0 + i);
  uint32_t low[kSegPerThread];
  seg_low_parts(s, table, tile, low);
#pragma unroll
  for (uint32_t k = 0; k < kSegPerThread; ++k) {
    const uint32_t x = threadIdx.x + k * kSegThreads;
    plane[x & 3u][x >> 2] = low[k];
  }
  __syncthreads();
  const uint32_t phase = (uint32_t)(reinterpret_cast<uintptr_t>(ms) >> 2) & 3u;
  const bool aligned = phase == ((uint32_t)reinterpret_cast<uintptr_t>(fe) & 3u);
  const uint32_t width = min(kSegTile, s.A - tile.x0), lane = threadIdx.x & 31u;
  // One warp per row: a row's set-up is shared by 16 vectors a lane.
  for (uint32_t i = threadIdx.x >> 5; i < tile.h1 - tile.h0; i += kSegThreads / 32u) {
    const uint32_t hi = high[i], from = (tile.h0 + i) * s.A + tile.x0;  // index of x = 0 of the tile
    if (from > s.last || from + width <= s.first) continue;
    const uint32_t b = from < s.first ? s.first - from : 0u, e = min(width, s.last - from + 1u);  // x in [b, e)
    const uint32_t at = from + b - s.first;  // output position of x = b
    uint32_t* const m = ms + at;
    uint8_t* const f = fe + at;
    uint32_t head = e - b, vectors = 0u;
    if (aligned) {
      head = min((0u - (at + phase)) & 3u, head);
      vectors = (e - b - head) / 4u;
    }
    uint4* const mv = reinterpret_cast<uint4*>(m + head);
    uint32_t* const fv = reinterpret_cast<uint32_t*>(f + head);
    const uint32_t* p[4];  // element c of vector v is p[c][v]: plane and offset are the same for the whole row
#pragma unroll
    for (uint32_t c = 0; c < 4; ++c) p[c] = plane[(b + head + c) & 3u] + ((b + head + c) >> 2);
#pragma unroll 4
    for (uint32_t v = lane; v < vectors; v += 32u) {
      uint32_t sum[4];
#pragma unroll
      for (uint32_t c = 0; c < 4; ++c) sum[c] = p[c][v] + hi;
      // A sum is infeasible when it reaches kSegInfeasible = 2^31 - 1: its top
      // bit after adding one.
      const uint32_t dead = ((sum[0] + 1u) >> 31) | ((sum[1] + 1u) >> 31 << 8) | ((sum[2] + 1u) >> 31 << 16) |
                            ((sum[3] + 1u) >> 31 << 24);
      __stcs(mv + v, make_uint4(seg_makespan(sum[0]), seg_makespan(sum[1]), seg_makespan(sum[2]), seg_makespan(sum[3])));
      __stcs(fv + v, dead ^ 0x01010101u);
    }
    // The elements before the first and after the last vector.
    const uint32_t single = e - b - 4u * vectors;
    for (uint32_t t = lane; t < single; t += 32u) {
      const uint32_t k = t < head ? t : t + 4u * vectors, x = b + k;
      const uint32_t sum = plane[x & 3u][x >> 2] + hi;
      m[k] = seg_makespan(sum);
      f[k] = sum < kSegInfeasible;
    }
  }
}

// Sums where the low parts do not fill a tile (A < kSegTile).  A block has the
// sums of all low parts and of the rows its kSegDirect mappings per thread lie
// in, in shared memory: each mapping is two lookups.
__global__ void __launch_bounds__(kSegThreads) segment_direct_kernel(const __grid_constant__ SegSums s,
                                                                     const uint32_t* table, uint32_t* ms,
                                                                     uint8_t* fe) {
  __shared__ uint32_t low[kSegTile], high[kSegThreads * kSegDirect / 3 + 2];
  cudaGridDependencySynchronize();
  const uint32_t from = s.first + blockIdx.x * (kSegThreads * kSegDirect);
  const uint32_t count = min(s.last - from + 1u, kSegThreads * kSegDirect);
  const uint32_t h0 = from / s.A, rows = (from + count - 1u) / s.A - h0 + 1u;  // A >= 3
  for (uint32_t i = threadIdx.x; i < s.A + rows; i += kSegThreads) {
    if (i < s.A) low[i] = segment_sum(s, table, 0u, s.split, i);
    else high[i - s.A] = segment_sum(s, table, s.split, s.count, h0 + i - s.A);
  }
  __syncthreads();
#pragma unroll
  for (uint32_t k = 0; k < kSegDirect; ++k) {
    const uint32_t i = k * kSegThreads + threadIdx.x;
    if (i >= count) continue;
    const uint32_t idx = from + i, h = idx / s.A, sum = low[idx - h * s.A] + high[h - h0];
    ms[idx - s.first] = seg_makespan(sum);
    fe[idx - s.first] = sum < kSegInfeasible;
  }
}

// Launch a sum kernel as a programmatic dependent of the tables' launch.
template <typename... Params, typename... Args>
cudaError_t launch_after_tables(void (*kernel)(Params...), uint32_t blocks, cudaStream_t st, Args... args) {
  cudaLaunchAttribute after{};
  after.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  after.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(kSegThreads);
  cfg.stream = st;
  cfg.attrs = &after;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Launch KERNEL<NC> over a plan's tables, NC by its largest segment.
#define BF_SEG_LAUNCH(KERNEL, BLOCKS, ...)                                                                       \
  do {                                                                                                           \
    static std::atomic<uint64_t> ready2{0}, ready3{0};                                                           \
    const bool two = plan.nmax <= kLtBatchTools;                                                                 \
    const size_t smem = sizeof(uint32_t) * lt_rows<false>(plan.nmax) * kSegThreads;                              \
    const size_t most = sizeof(uint32_t) * lt_rows<false>(two ? kLtBatchTools : kSegMaxTools) * kSegThreads;     \
    const cudaError_t e = two ? allow_dyn_smem(KERNEL<2>, most, &ready2) : allow_dyn_smem(KERNEL<3>, most, &ready3); \
    if (e != cudaSuccess) return e;                                                                              \
    if (two) KERNEL<2><<<(BLOCKS), kSegThreads, smem, st>>>(__VA_ARGS__);                                        \
    else KERNEL<3><<<(BLOCKS), kSegThreads, smem, st>>>(__VA_ARGS__);                                            \
    return cudaGetLastError();                                                                                   \
  } while (0)

}  // namespace

cudaError_t launch_segment_tables(const SegPlan& plan, uint32_t* table, cudaStream_t st) {
  if (plan.tables == 0u) return cudaSuccess;
  BF_SEG_LAUNCH(segment_table_kernel, plan.first_block[plan.tables], plan, table);
}

cudaError_t launch_segment_optimum(const SegPlan& plan, uint32_t radix, SegSync* sync, BestRecord* host_best,
                                   cudaStream_t st) {
  BF_SEG_LAUNCH(segment_optimum_kernel, plan.tables ? plan.first_block[plan.tables] : 1u, plan, radix, sync, host_best);
}

cudaError_t launch_segment_eval(const SegSums& sums, const uint32_t* table, uint32_t* ms, uint8_t* fe,
                                cudaStream_t st) {
  if (sums.x_tiles) {
    const uint32_t blocks = sums.x_tiles * ((sums.h_hi - sums.h_lo) / sums.rows + 1u);
    return launch_after_tables(segment_eval_kernel, blocks, st, sums, table, ms, fe);
  }
  const uint32_t blocks = (sums.last - sums.first) / (kSegThreads * kSegDirect) + 1u;
  return launch_after_tables(segment_direct_kernel, blocks, st, sums, table, ms, fe);
}

}  // namespace bfk
