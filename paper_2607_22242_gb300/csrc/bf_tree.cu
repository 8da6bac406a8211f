// bf_tree.cu -- kernels of the tree search (bf_tree.cuh).  All state is 32 slots
// wide.
//
//   tree_bound_kernel  : the starting bound from the scored candidates.
//   tree_start_kernel  : one thread per combination of the first d0 tools'
//                        modes, simulated from time 0, bounded and appended to
//                        level d0 (one launch instead of d0 small ones).
//   tree_expand_kernel : one thread per (parent, mode of the next tool); the
//                        child is resumed to its checkpoint, bounded, and the
//                        survivors are appended to the next level's buffer
//                        (one atomicAdd per warp on the level's count).
//   tree_leaf_kernel   : one warp per 32 leaf-level nodes (one per lane) and a
//                        part of the combinations of the last D tools' modes,
//                        walked over the leaf window (tools from the
//                        lowest one that can still be running at a leaf
//                        checkpoint; compiled for 8..32 slots), without those
//                        in which a leaf tool must end too late for the bound
//                        the launch began with; per-block best (makespan, index)
//                        merged into one 16-byte record by compare-and-swap.
//
// Level sizes stay on the device: the launches of a chain of levels are sized
// for the most nodes a level can hold and read how many there are.
#include <cuda_runtime.h>

#include "bf_launch.h"
#include "bf_plan.h"
#include "bf_tree.h"

namespace bfk {
namespace {

constexpr int kTreeThreads = 256;
constexpr int kTreeWarps = kTreeThreads / 32;
constexpr int kNW = NodeWords<kTreeSlots>::value;

__device__ __forceinline__ uint32_t read_count(const uint32_t* count) {
  return *reinterpret_cast<const volatile uint32_t*>(count);
}

__global__ void tree_bound_kernel(const uint32_t* ms, const uint8_t* fe, uint32_t n, TreeBounds* bounds,
                                  TreeCounters* ctr) {
  uint32_t b = kInfeasible;
  for (uint32_t j = 0; j < n; ++j)
    if (fe[j] == 1u && ms[j] < b) b = ms[j];
  bounds->live = b;
  ctr->incumbent = b;
}

// The bound of the coming leaf launch (TreeBounds::leaf).
__device__ __forceinline__ void note_leaf_bound(TreeBounds* bounds) {
  if (blockIdx.x == 0u && threadIdx.x == 0u) bounds->leaf = read_bound(&bounds->live);
}

// Append this lane's node (if it keeps one) to a level: a slot per lane from
// one atomicAdd per warp.
__device__ __forceinline__ void append_node(bool keep, const State<kTreeSlots>& s, Digits dg, TreeLevel dst,
                                            uint32_t cap, TreeCounters* ctr) {
  const uint32_t ballot = __ballot_sync(0xFFFFFFFFu, keep);
  if (ballot == 0u) return;
  const uint32_t lane = threadIdx.x & 31u, leader = __ffs(ballot) - 1;
  uint32_t base = 0u;
  if (lane == leader) {
    base = atomicAdd(dst.count, (uint32_t)__popc(ballot));
    atomicAdd(&ctr->nodes, (unsigned long long)__popc(ballot));
  }
  base = __shfl_sync(0xFFFFFFFFu, base, leader);
  if (!keep) return;
  const uint32_t slot = base + __popc(ballot & ((1u << lane) - 1u));
  if (slot >= cap) {  // cannot happen (nodes * radix <= cap); recorded, never written
    atomicOr(&ctr->error, 1u);
    return;
  }
  store_node(s, dg, dst.buf, cap, slot);
}

__global__ void __launch_bounds__(kTreeThreads, 2) tree_start_kernel(
    const __grid_constant__ TablesW tb, const __grid_constant__ TreeConsts tc, uint32_t d0, uint32_t combos,
    TreeLevel dst, uint32_t cap, TreeBounds* bounds, TreeCounters* ctr) {
  __shared__ SmemTablesW sd;
  __shared__ uint32_t rt[ReadyTable<kTreeSlots>::size];
  __shared__ uint32_t ef[kTreeSlots * kTreeThreads];  // forward_bound scratch, [tool][thread]
  note_leaf_bound(bounds);
  load_smem_tables(tb, sd);
  fill_ready_table<kTreeSlots>(tb, rt);
  __syncthreads();
  const uint32_t p = blockIdx.x * kTreeThreads + threadIdx.x;
  State<kTreeSlots> s;
  Digits dg{0u, 0u};
  bool keep = false;
  if (p < combos) {
    dg = leaf_digits(p, tc.radix, d0, 0u);
    init_state(s, tb.all_mask);
    keep = expand_start<kTreeSlots>(tb, sd, rt, tc, s, dg, d0, read_bound(&bounds->live), ef + threadIdx.x, kTreeThreads);
  }
  append_node(keep, s, dg, dst, cap, ctr);
}

__global__ void __launch_bounds__(kTreeThreads, 2) tree_expand_kernel(
    const __grid_constant__ TablesW tb, const __grid_constant__ TreeConsts tc, TreeLevel src, uint32_t pop, uint32_t d,
    TreeLevel dst, uint32_t cap, TreeBounds* bounds, TreeCounters* ctr) {
  __shared__ SmemTablesW sd;
  __shared__ uint32_t rt[ReadyTable<kTreeSlots>::size];
  __shared__ uint32_t ef[kTreeSlots * kTreeThreads];  // forward_bound scratch, [tool][thread]
  note_leaf_bound(bounds);
  // Thread t: mode a = t / cnt of tool d for parent lo + t % cnt, so that a
  // warp's lanes hold neighbouring parents with the same new mode.
  const uint32_t size = read_count(src.count), cnt = min(size, pop), lo = size - cnt;
  if (blockIdx.x * kTreeThreads >= cnt * tc.radix) return;
  load_smem_tables(tb, sd);
  fill_ready_table<kTreeSlots>(tb, rt);
  __syncthreads();
  const uint32_t t = blockIdx.x * kTreeThreads + threadIdx.x;
  const uint32_t a = t / cnt, j = t - a * cnt;
  bool keep = false;
  State<kTreeSlots> s;
  Digits dg{0u, 0u};
  if (a < tc.radix) {
    load_node(src.buf, cap, lo + j, s, dg);
    keep = expand_child<kTreeSlots>(tb, sd, rt, tc, s, dg, d, a, read_bound(&bounds->live), ef + threadIdx.x, kTreeThreads);
  }
  append_node(keep, s, dg, dst, cap, ctr);
}

// Lexicographic (makespan, index) minimum of the 16-byte record at *p.  Every
// failed compare-and-swap means another block stored a smaller record, so the
// loop ends; it is bounded all the same and reports if it ever gave up.
__device__ void best_min(BestRecord* p, uint64_t ms, uint64_t idx, TreeCounters* ctr) {
  BestRecord cur = *p;
  for (int it = 0; it < 4096; ++it) {
    if (cur.ms < ms || (cur.ms == ms && cur.idx <= idx)) return;
    const BestRecord want{ms, idx};
    const BestRecord old = atomicCAS(p, cur, want);
    if (old.ms == cur.ms && old.idx == cur.idx) return;
    cur = old;
  }
  atomicOr(&ctr->error, 2u);
}

__device__ __forceinline__ LaneBest shfl_best(const LaneBest& b, int o) {
  LaneBest r;
  r.ms = __shfl_xor_sync(0xFFFFFFFFu, b.ms, o);
  r.dg.now = __shfl_xor_sync(0xFFFFFFFFu, b.dg.now, o);
  r.dg.que = __shfl_xor_sync(0xFFFFFFFFu, b.dg.que, o);
  return r;
}

// Leaf kernel over a window of NW slots (tools [W0, W0 + NW)).
// Block shape of the leaf kernel per window width: 256 threads for narrow
// windows, 128 for wide ones (their registers and per-lane shared state leave
// room for more small blocks than large ones: 20 warps/SM instead of 16 at
// 24 slots; measured 10-20 % faster there).
template <int NW>
struct LeafShape {
  static constexpr int threads = NW >= 16 ? 128 : 256;
  static constexpr int warps = threads / 32;
  static constexpr int min_blocks = NW <= 12 ? 4 : NW <= 16 ? 6 : NW <= 24 ? 5 : 4;
};

// The tasks of the leaf kernel (leaf_task).  About kTreeLeafTasks tasks over all
// nodes (each prepares its nodes anew; a quarter as many take as long, within 4 %
// over 12 DAGs), at least 16 combinations each, taken in turn by the grid's warps.
// Few nodes are cut finer, down to 2 combinations a task, for about kTreeLeafFill
// tasks: one warp for each place on the GPU in the 20- and 24-slot forms (5 blocks
// of 4 warps on each of 152 SMs; up to 12 slots there are 32 places per SM, at 16
// slots 24, at 32 slots 16), which otherwise waits for a chain of 16 simulations
// on an eighth of them.  Full / binary space without and with it: 8 tools 0.18 ->
// 0.085 / 0.09 -> 0.08 ms, 14 layered tools 0.46 -> 0.28 / 0.27 -> 0.11, 16 tools
// 0.67 -> 0.51 / 0.33 -> 0.12, 18 tools 0.85 -> 0.59 / 0.35 -> 0.14, 20 tools 0.97
// -> 0.76 / 0.38 -> 0.18.
constexpr uint32_t kTreeLeafTasks = 16384;
constexpr uint32_t kTreeLeafFill = 3072;

template <int NW>
__global__ void __launch_bounds__(LeafShape<NW>::threads, LeafShape<NW>::min_blocks) tree_leaf_kernel(
    const __grid_constant__ TablesW tb, const __grid_constant__ TablesT<NW> tw, const __grid_constant__ TreeConsts tc,
    TreeLevel src, uint32_t cap, TreeBounds* bounds, BestRecord* best, TreeCounters* ctr) {
  extern __shared__ uint32_t lane_state[];
  __shared__ SmemTablesT<NW> sdw;
  __shared__ uint32_t rtw[ReadyTable<NW>::size];
  __shared__ uint32_t wb_ms[LeafShape<NW>::warps], wb_now[LeafShape<NW>::warps], wb_que[LeafShape<NW>::warps];
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint32_t cnt = read_count(src.count), groups = (cnt + 31u) / 32u;
  // With a lone last tool, combinations cover the leaf tools but the last
  // one, each standing for radix mappings.
  const uint32_t ncomb = tc.alone_last ? tc.combos / tc.radix : tc.combos;
  const uint32_t per = max(groups, 1u);
  const uint32_t want = max(max(1u, min((kTreeLeafTasks + groups - 1u) / per, (ncomb + 15u) / 16u)),
                            min(kTreeLeafFill / per, (ncomb + 1u) / 2u));
  const uint32_t chunk = (ncomb + want - 1u) / want, parts = (ncomb + chunk - 1u) / chunk;
  if (blockIdx.x * LeafShape<NW>::warps >= groups * parts) return;
  load_smem_tables(tw, sdw);
  fill_ready_table<NW>(tw, rtw);
  __syncthreads();
  LaneBest lb;
  uint32_t* const slot = lane_state + threadIdx.x;
  for (uint32_t task = blockIdx.x * LeafShape<NW>::warps + warp; task < groups * parts;
       task += gridDim.x * LeafShape<NW>::warps) {
    uint32_t nodes;
    const uint32_t ran = leaf_task<NW, LeafShape<NW>::threads>(tb, tw, sdw, rtw, tc, src.buf, cap, cnt, task / parts,
                                                               task % parts, parts, chunk, bounds, slot, lb, &nodes);
    if (nodes == 0u) continue;
    const uint32_t all = __reduce_add_sync(0xFFFFFFFFu, ran);
    if (lane == 0) {
      if (task % parts == 0) atomicAdd(&ctr->leaf_nodes, (unsigned long long)__popc(nodes));
      if (all) atomicAdd(&ctr->leaves, (unsigned long long)all * (tc.alone_last ? tc.radix : 1u));
    }
  }
  // warp, then block minimum; one record update per block
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const LaneBest other = shfl_best(lb, o);
    lb.offer(other.ms, other.dg, tc.tie_pow3());
  }
  if (lane == 0) {
    wb_ms[warp] = lb.ms;
    wb_now[warp] = lb.dg.now;
    wb_que[warp] = lb.dg.que;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    LaneBest b;
    for (int w = 0; w < LeafShape<NW>::warps; ++w) b.offer(wb_ms[w], Digits{wb_now[w], wb_que[w]}, tc.tie_pow3());
    if (b.ms != kInfeasible) {
      atomicMin(&bounds->live, b.ms);
      best_min(best, b.ms, index_of(b.dg, tc.pow3), ctr);
    }
  }
}

}  // namespace

size_t tree_node_words() { return (size_t)kNW; }

cudaError_t launch_tree_bound(const uint32_t* ms, const uint8_t* fe, uint32_t n, TreeBounds* bounds, TreeCounters* ctr,
                              cudaStream_t st) {
  tree_bound_kernel<<<1, 1, 0, st>>>(ms, fe, n, bounds, ctr);
  return cudaGetLastError();
}

cudaError_t launch_tree_start(const TablesW& tb, const TreeConsts& tc, uint32_t d0, TreeLevel dst, uint32_t cap,
                              TreeBounds* bounds, TreeCounters* ctr, cudaStream_t st) {
  uint32_t combos = 1;
  for (uint32_t i = 0; i < d0; ++i) combos *= tc.radix;
  tree_start_kernel<<<(combos + kTreeThreads - 1) / kTreeThreads, kTreeThreads, 0, st>>>(tb, tc, d0, combos, dst, cap,
                                                                                         bounds, ctr);
  return cudaGetLastError();
}

cudaError_t launch_tree_expand(const TablesW& tb, const TreeConsts& tc, TreeLevel src, uint32_t pop,
                               uint32_t most_nodes, uint32_t d, TreeLevel dst, uint32_t cap, TreeBounds* bounds,
                               TreeCounters* ctr, cudaStream_t st) {
  const uint64_t threads = (uint64_t)(most_nodes < pop ? most_nodes : pop) * tc.radix;
  const unsigned grid = (unsigned)((threads + kTreeThreads - 1) / kTreeThreads);
  tree_expand_kernel<<<grid, kTreeThreads, 0, st>>>(tb, tc, src, pop, d, dst, cap, bounds, ctr);
  return cudaGetLastError();
}

template <int NW>
static cudaError_t leaf_launch(const TablesW& tb, const TreeConsts& tc, TreeLevel src, uint32_t cap,
                               uint32_t most_nodes, TreeBounds* bounds, BestRecord* best, TreeCounters* ctr,
                               cudaStream_t st) {
  static std::atomic<uint64_t> ready{0};
  const size_t smem = sizeof(uint32_t) * LaneWords<NW>::value * LeafShape<NW>::threads;
  cudaError_t e = allow_dyn_smem(tree_leaf_kernel<NW>, smem, &ready);
  int dev = 0, sms = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  TablesT<NW> tw;
  host::build_window(tb, tc.W0, &tw);
  // At most this many tasks (see the kernel), and a few waves of the GPU.
  const uint64_t groups = (most_nodes + 31u) / 32u, tasks = kTreeLeafTasks + groups;
  const uint64_t need = (tasks + LeafShape<NW>::warps - 1) / LeafShape<NW>::warps;
  const uint64_t most = (uint64_t)sms * LeafShape<NW>::min_blocks * 8u;
  tree_leaf_kernel<NW><<<(unsigned)(need < most ? need : most), LeafShape<NW>::threads, smem, st>>>(
      tb, tw, tc, src, cap, bounds, best, ctr);
  return cudaGetLastError();
}

cudaError_t launch_tree_leaf(const TablesW& tb, const TreeConsts& tc, TreeLevel src, uint32_t cap,
                             uint32_t most_nodes, TreeBounds* bounds, BestRecord* best, TreeCounters* ctr,
                             cudaStream_t st) {
  const uint32_t nw = tb.n - tc.W0;
#define BF_TRY(NW) \
  if (nw <= (uint32_t)NW) return leaf_launch<NW>(tb, tc, src, cap, most_nodes, bounds, best, ctr, st);
  BF_TREE_BUCKETS(BF_TRY)
#undef BF_TRY
  return cudaErrorInvalidValue;
}

}  // namespace bfk
