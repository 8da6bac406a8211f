// bf_capi_tree.cu -- bf_search_tree (include/bf.h): the host side of the tree
// search, whose kernels are in bf_tree.cu.  The host decides which level to pop
// next and launches a chain of expansions down to the leaves; it waits (bounded)
// once per chain, for how many nodes each level has kept.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <cstring>
#include <new>
#include <chrono>
#include <vector>

#include "bf_capi_internal.h"

using namespace bfcapi;
using bfk::host::pow3;

namespace {

// The tree search's record, bound, counters and level sizes, copied together.
constexpr size_t kTreeStateBytes = offsetof(bf_scratch, idx) - offsetof(bf_scratch, best);

int search_tree_impl(const bf_scenario* scn_const, uint32_t space, uint32_t flags, uint64_t hint_index,
                     bf_result* out, bf_tree_stats* stats, void* cuda_stream) {
  const char* who = "bf_search_tree";
  if (!scn_const || !out) return fail(BF_EINVAL, "%s: NULL argument", who);
  if (space != BF_SPACE_BINARY && space != BF_SPACE_FULL)
    return fail(BF_EINVAL, "%s: space %u is neither BF_SPACE_BINARY (2) nor BF_SPACE_FULL (3)", who, space);
  if (flags & ~(uint32_t)BF_TREE_NO_PRUNE) return fail(BF_EINVAL, "%s: unknown flags 0x%x", who, flags);
  if (const int rc = check_device(scn_const, who)) return rc;
  if (scn_const->seg.count && !(flags & BF_TREE_NO_PRUNE)) {
    // Every segment between two barriers is small enough to be enumerated on
    // its own (bf_segments.cuh): a 32-tool spine with fan-outs 1.58 ms
    // -> 41 us a call, either space.
    const int rc = segment_optimum(scn_const, space, out, static_cast<cudaStream_t>(cuda_stream), who);
    if (rc == BF_OK && stats) {
      std::memset(stats, 0, sizeof *stats);
      const bfk::SegPlan& seg = scn_const->seg;
      stats->nodes = stats->leaf_nodes = seg.count;
      for (uint32_t j = 0; j < seg.count; ++j) {
        uint64_t mappings = 1;
        for (uint32_t v = seg.start[j]; v < seg.start[j + 1]; ++v) mappings *= space;
        stats->leaves += mappings;
      }
      stats->launches = 1;
      stats->leaf_depth = seg.nmax;
      stats->incumbent_us = 0xFFFFFFFFu;
    }
    return rc;
  }
  // The handle's lazily allocated level buffers are scratch, not state.
  bf_scenario* scn = const_cast<bf_scenario*>(scn_const);
  // The tree runs on the tools renumbered with the sources first
  // (relabel_sources_first): a source in a later layer is then decided near
  // the root instead of keeping every node's window open from time 0, and the
  // model's results do not change.  Indices stay canonical: slot v holds tool
  // tb.orig[v], whose digit weighs 3^orig[v].
  bfk::TablesW renumbered;
  const bool relabeled = bfk::host::relabel_sources_first(scn->wide, &renumbered);
  const bfk::TablesW& tb = relabeled ? renumbered : scn->wide;
  const uint32_t n = scn->desc.n, R = space;
  const bool prune = !(flags & BF_TREE_NO_PRUNE);
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);

  // Constants: the leaf depth, the bound's per-tool durations, digit powers.
  bfk::TreeConsts tc;
  bfk::host::tree_consts(tb, R, prune, &tc);

  // Level buffers: level d holds up to R * kPop nodes (one pop of its parent
  // level); nodes are popped from the deepest non-empty level, so no level
  // ever holds more.
  constexpr uint32_t kPop = 65536;
  const uint32_t cap = R * kPop;
  const uint32_t levels = tc.leaf_level + 1;
  const size_t level_words = bfk::tree_node_words() * cap;
  const size_t need = sizeof(uint32_t) * level_words * levels;
  cudaError_t e = cudaSuccess;
  if (scn->levels_bytes < need) {
    if (scn->d_levels) cudaFree(scn->d_levels);
    scn->d_levels = nullptr;
    scn->levels_bytes = 0;
    e = lib_malloc(reinterpret_cast<void**>(&scn->d_levels), need);
    if (e != cudaSuccess) return cuda_fail(e, who);
    scn->levels_bytes = need;
  }

  auto tree_level = [&](uint32_t d) { return bfk::TreeLevel{scn->d_levels + level_words * d, scn->d_scratch->count + d}; };

  bf_scratch* h = scn->h_scratch;
  bf_scratch* dv = scn->d_scratch;
  uint32_t launches = 0;
  begin_call(scn);

  // 1. Reset the record, bound, counters and level sizes (pinned, and not
  //    written again before the first wait below).
  h->best.ms = ~0ull;
  h->best.idx = ~0ull;
  h->bounds.live = h->bounds.leaf = 0xFFFFFFFFu;
  std::memset(&h->ctr, 0, sizeof h->ctr);
  h->ctr.incumbent = 0xFFFFFFFFu;
  std::memset(h->count, 0, sizeof h->count);
  e = cudaMemcpyAsync(&dv->best, &h->best, kTreeStateBytes, cudaMemcpyHostToDevice, st);

  // 2. Incumbent: the best feasible of a few mappings of the space (the hint
  //    if it lies in it, all-cpu, all-gpu_now, each tool on its isolated-faster
  //    device, and all-gpu_queue in the full space), scored and compared on the
  //    device.
  if (prune && e == cudaSuccess) {
    const uint64_t total = pow3(n);
    uint32_t nc = 0;
    bool hint_ok = hint_index < total;
    if (hint_ok && R == 2)
      for (uint64_t v = hint_index; v; v /= 3) hint_ok = hint_ok && (v % 3 != 2);
    if (hint_ok) h->idx[nc++] = hint_index;
    const bfk::TablesW& tsc = scn->wide;  // the scenario's numbering
    uint64_t now = 0, fast = 0, p = 1;
    for (uint32_t i = 0; i < n; ++i, p *= 3) {
      now += p;
      if ((tsc.wnow[i] >> 10) < tsc.cpu[i]) fast += p;
    }
    h->idx[nc++] = 0;
    h->idx[nc++] = now;
    h->idx[nc++] = fast;
    if (R == 3) h->idx[nc++] = 2 * now;
    e = launch_list(scn, scn->d_host_scratch->idx, nc, dv->ms, dv->fe, st);
    if (e == cudaSuccess) e = bfk::launch_tree_bound(dv->ms, dv->fe, nc, &dv->bounds, &dv->ctr, st);
    launches += 2;
  }
  if (e != cudaSuccess) return cuda_fail(e, who);

  // 3. Depth first over levels, in chains of launches that the host does not
  //    wait between: from the deepest level that holds nodes, up to `pop` nodes
  //    of it are expanded into the next level, up to `pop` of those (all of the
  //    leaf level) into the one after, and so on to the leaves; after the
  //    chain the host reads how many nodes each level has kept.  The levels
  //    below the one a chain starts from are empty.  The first chain starts
  //    with every combination of the first d0 tools.  A tree of more
  //    leaf-level nodes than the start makes begins with two dives, chains of
  //    kDives[i] nodes per level, whose leaves set the bound; their other nodes
  //    are then dropped and the search starts over with that bound.  Over both
  //    spaces of 12 layered and sparse DAGs of 8 to 26 tools (geometric mean of the
  //    calls): dives of {256, 2048} nodes 0.29 ms, {256} 0.36, {1024} 0.38, {8192}
  //    0.45.  Dives also pay below kPop leaf-level nodes (14 layered tools
  //    0.60 -> 0.28 ms, 14 sparse ones 0.46 -> 0.28, the binary space of 24 tools 2.4
  //    -> 0.59).
  //    With these chains, the leaf modes (bf_tree.cuh node_leaf_modes) and the
  //    leaf kernel's tasks full searches went from 2.30 to 0.59 ms (18 layered
  //    tools), 4.06 to 0.76 (20), 7.4 to about 1.5 (24) and 6.4 to 1.4 ms (26).
  static constexpr uint32_t kDives[] = {256, 2048};
  constexpr uint32_t kStart = 8192;
  // The whole search, not only each wait, is held to the wait limit.
  const auto t_start = std::chrono::steady_clock::now();
  const uint32_t limit_ms = wait_limit_ms();
  uint32_t d0 = 0;
  uint64_t start_nodes = 1, leaf_level_nodes = 1;  // radix^d0; radix^L, saturating
  while (d0 < tc.leaf_level && start_nodes * R <= kStart) {
    start_nodes *= R;
    ++d0;
  }
  for (uint32_t i = 0; i < tc.leaf_level && leaf_level_nodes <= kStart; ++i) leaf_level_nodes *= R;
  auto chain = [&](uint32_t from, uint64_t most, uint32_t pop) {  // most: nodes level `from` may hold
    for (uint32_t d = from; d < tc.leaf_level && e == cudaSuccess; ++d) {
      e = bfk::launch_tree_expand(tb, tc, tree_level(d), pop, (uint32_t)most, d, tree_level(d + 1), cap, &dv->bounds,
                                  &dv->ctr, st);
      most = (most < pop ? most : pop) * R;
      ++launches;
    }
    if (e == cudaSuccess)
      e = bfk::launch_tree_leaf(tb, tc, tree_level(tc.leaf_level), cap, (uint32_t)most, &dv->bounds, &dv->best,
                                &dv->ctr, st);
    ++launches;
  };
  auto start = [&]() {
    e = bfk::launch_tree_start(tb, tc, d0, tree_level(d0), cap, &dv->bounds, &dv->ctr, st);
    ++launches;
  };
  start();
  if (prune && leaf_level_nodes > kStart && e == cudaSuccess) {
    for (const uint32_t pop : kDives) {
      if (e == cudaSuccess) chain(d0, start_nodes, pop);
      if (e == cudaSuccess) e = cudaMemsetAsync(dv->count, 0, sizeof dv->count, st);
      if (e == cudaSuccess) start();
    }
  }
  std::vector<uint32_t> size(levels, 0);
  uint32_t from = d0;
  uint64_t most = start_nodes;
  for (;;) {
    if (e == cudaSuccess) chain(from, most, kPop);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(h->count, dv->count, sizeof h->count, cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return cuda_fail(e, who);
    const int rc = wait_stream(st, who);
    if (rc != BF_OK) return rc;
    // What each level of the chain has kept: all but the last kPop nodes.
    for (uint32_t d = from; d < tc.leaf_level; ++d) size[d] = h->count[d] > kPop ? h->count[d] - kPop : 0u;
    int d = (int)tc.leaf_level - 1;
    while (d >= 0 && size[d] == 0) --d;
    if (d < 0) break;
    if (limit_ms) {
      const auto ms = std::chrono::duration_cast<std::chrono::milliseconds>(std::chrono::steady_clock::now() - t_start);
      if (ms.count() > (long long)limit_ms)
        return fail(BF_ETIMEOUT, "%s: search not finished after %u ms", who, limit_ms);
    }
    from = (uint32_t)d;
    most = size[d];
    for (uint32_t i = 0; i < levels; ++i) h->count[i] = i <= from ? size[i] : 0u;
    e = cudaMemcpyAsync(dv->count, h->count, sizeof h->count, cudaMemcpyHostToDevice, st);
  }

  // 4. The record.
  e = cudaMemcpyAsync(&h->best, &dv->best, kTreeStateBytes, cudaMemcpyDeviceToHost, st);
  if (e != cudaSuccess) return cuda_fail(e, who);
  const int rc = end_call(scn, st, who);
  if (rc != BF_OK) return rc;
  if (h->ctr.error) return fail(BF_ECUDA, "%s: internal error 0x%x in the tree kernels", who, h->ctr.error);
  fill_best(h->best, n, out);
  if (stats) {
    stats->nodes = 1 + h->ctr.nodes;
    stats->leaf_nodes = h->ctr.leaf_nodes;
    stats->leaves = h->ctr.leaves;
    stats->launches = launches;
    stats->leaf_depth = tc.D;
    stats->incumbent_us = h->ctr.incumbent;
  }
  return BF_OK;
}

}  // namespace

extern "C" {

// Host allocation failures and other C++ exceptions stay inside the library.
int bf_search_tree(const bf_scenario* scn, uint32_t space, uint32_t flags, uint64_t hint_index, bf_result* out,
                   bf_tree_stats* stats, void* cuda_stream) {
  try {
    return search_tree_impl(scn, space, flags, hint_index, out, stats, cuda_stream);
  } catch (const std::bad_alloc&) {
    return fail(BF_ENOMEM, "bf_search_tree: host allocation failed");
  } catch (const std::exception& ex) {
    return fail(BF_EINVAL, "bf_search_tree: %s", ex.what());
  }
}

}  // extern "C"
