// Host build of the tree search's node logic (bf_tree.cuh, with bf_plan.h and
// bf_sim.cuh), for tests that run without a GPU: the same constants
// (host::tree_consts), the same sources-first renumbering, the start from the
// first tools' modes (expand_start), node expansion with its bound
// (expand_child), the leaf tools' modes within the bound (node_leaf_modes,
// leaf_mode_combos, leaf_mode_digits), the leaf window (node_to_window), the
// leaf runs (leaf_run; leaf_combos unpruned) and the tie rule (LaneBest), walked
// depth first on one CPU thread, one node at a time (the tasks of a warp, which
// share nodes, are run by host_warp.cpp).  Pruning is strict, so any order of
// the nodes gives the same optimum as the kernels' breadth-first levels.  Test
// infrastructure only; the library never runs this.
#include <algorithm>
#include <cstdint>
#include <cstring>
#include <vector>

#define __device__
#define __host__
#define __forceinline__ inline
using std::max;
using std::min;
static inline int __popc(unsigned x) { return __builtin_popcount(x); }
static inline int __ffs(unsigned x) { return __builtin_ffs((int)x); }
static inline int __clz(unsigned x) { return x ? __builtin_clz(x) : 32; }
static inline unsigned long long __umul64hi(unsigned long long a, unsigned long long b) {
  return (unsigned long long)(((unsigned __int128)a * b) >> 64);
}

#include "host_warp.h"

#include "../paper_2607_22242_gb300/csrc/bf_tree.cuh"

using namespace bfk;

namespace {

template <int NW>
struct Search {
  const TablesW& tb;
  const TreeConsts& tc;
  SmemTablesW sd;
  std::vector<uint32_t> rt;
  TablesT<NW> tw;
  SmemTablesT<NW> sdw;
  std::vector<uint32_t> rtw, ef, node, slot;
  uint32_t bound;
  unsigned long long best_ms = ~0ull, best_idx = ~0ull, nodes = 0, leaves = 0;
  // Leaf nodes are reduced as the leaf kernel reduces its lanes: 32
  // consecutive ones through LaneBest::offer (the warp's shuffle tree and
  // the block's loop), then into the record by canonical index.
  LaneBest group;
  uint32_t in_group = 0;

  Search(const TablesW& t, const TreeConsts& c, uint32_t b)
      : tb(t), tc(c), rt(ReadyTable<kTreeSlots>::size), rtw(ReadyTable<NW>::size), ef(kTreeSlots),
        node(NodeWords<kTreeSlots>::value), slot(LaneWords<NW>::value), bound(b) {
    threadIdx.x = 0;
    load_smem_tables(tb, sd);
    fill_ready_table<kTreeSlots>(tb, rt.data());
    host::build_window(tb, tc.W0, &tw);
    load_smem_tables(tw, sdw);
    fill_ready_table<NW>(tw, rtw.data());
  }

  // A leaf-level node: every combination of the leaf tools' modes that the
  // current bound leaves, or unpruned all of them (one node per "lane").
  void leaf(const State<kTreeSlots>& s, Digits dg) {
    store_node(s, dg, node.data(), 1u, 0u);
    LeafModes modes;
    if (tc.prune && !node_leaf_modes(node.data(), 1u, 0u, tb, tc, dg, bound, slot.data(), 1u, &modes)) return;
    node_to_window<NW>(node.data(), 1u, 0u, tc.W0, tw.n, slot.data(), 1u);
    const uint32_t each = tc.alone_last ? tc.radix : 1u;
    LaneBest lb;
    if (tc.prune) {
      const uint32_t combos = leaf_mode_combos(modes, tc);
      for (uint32_t k = 0; k < combos; ++k)
        leaves += leaf_run<NW, true>(tw, sdw, rtw.data(), tc, slot.data(), 1u, dg, leaf_mode_digits(modes, tc, k), lb, bound)
                      ? each : 0u;
    } else {
      leaves += each * leaf_combos<NW>(tw, sdw, rtw.data(), tc, slot.data(), 1u, dg, true, 0u, tc.combos / each, lb);
    }
    group.offer(lb.ms, lb.dg, tc.tie_pow3());
    if (++in_group == 32u) flush();
  }

  void flush() {
    const LaneBest b = group;
    group = LaneBest{};
    in_group = 0;
    if (b.ms == kInfeasible) return;
    bound = min(bound, b.ms);
    const unsigned long long idx = index_of(b.dg, tc.pow3);
    if (b.ms < best_ms || (b.ms == best_ms && idx < best_idx)) {
      best_ms = b.ms;
      best_idx = idx;
    }
  }

  void visit(const State<kTreeSlots>& s, Digits dg, uint32_t d) {
    ++nodes;
    if (d == tc.leaf_level) {
      leaf(s, dg);
      return;
    }
    for (uint32_t a = 0; a < tc.radix; ++a) {
      State<kTreeSlots> c = s;
      Digits cd = dg;
      if (expand_child<kTreeSlots>(tb, sd, rt.data(), tc, c, cd, d, a, bound, ef.data(), 1u)) visit(c, cd, d + 1);
    }
  }
};

template <int NW>
void run_search(const TablesW& tb, const TreeConsts& tc, uint32_t bound, uint32_t d0, unsigned long long* out) {
  Search<NW> sr(tb, tc, bound);
  uint32_t combos = 1;
  for (uint32_t i = 0; i < d0; ++i) combos *= tc.radix;
  for (uint32_t p = 0; p < combos; ++p) {
    State<kTreeSlots> s;
    init_state(s, tb.all_mask);
    const Digits dg = leaf_digits(p, tc.radix, d0, 0u);
    if (d0 == 0u || expand_start<kTreeSlots>(tb, sr.sd, sr.rt.data(), tc, s, dg, d0, sr.bound, sr.ef.data(), 1u))
      sr.visit(s, dg, d0);
  }
  sr.flush();
  out[0] = sr.best_ms;
  out[1] = sr.best_idx;
  out[2] = sr.nodes;
  out[3] = sr.leaves;
}

}  // namespace

// bf_search_tree's search over the space of radix `space` (2 or 3), starting
// from the incumbent makespan `bound` (0xFFFFFFFF: none), pruned or not, its
// nodes the expansions of all modes of the first min(d0, leaf level) tools.
// out[0..5] = best makespan (~0: none), its canonical index, nodes visited,
// leaf mappings simulated, renumbered (0/1), the leaf window width.
extern "C" int host_tree(const bf_scenario_desc* d, uint32_t space, uint32_t prune, uint32_t bound,
                         uint32_t d0, unsigned long long* out) {
  if (d->n < 1 || d->n > 32 || (space != 2 && space != 3)) return -1;
  TablesW t0, rt;
  host::build_tables(d, &t0);
  const bool relabeled = host::relabel_sources_first(t0, &rt);
  const TablesW& tb = relabeled ? rt : t0;
  TreeConsts tc;
  host::tree_consts(tb, space, prune != 0u, &tc);
  const uint32_t nw = tb.n - tc.W0;
  out[4] = relabeled ? 1u : 0u;
#define BF_TRY(NW)                                                               \
  if (nw <= (uint32_t)NW) {                                                      \
    out[5] = NW;                                                                 \
    run_search<NW>(tb, tc, bound, d0 < tc.leaf_level ? d0 : tc.leaf_level, out); \
    return 0;                                                                    \
  }
  BF_TREE_BUCKETS(BF_TRY)
#undef BF_TRY
  return -1;
}

// How many steps with a GPU tool running the unpruned leaf enumeration takes
// (leaf_combos), over every leaf node: with one LaneBest for all of a node's
// combinations as a lane has it, or (`fresh`) with a new one for each.
namespace {
struct Counted {  // reads of the slowdown table, one per such step
  const uint32_t* p;
  uint64_t* reads;
  uint32_t operator[](uint32_t k) const { ++*reads; return p[k]; }
};
template <int NW>
struct CountedTables {
  Counted f;
  const uint64_t* recip;
  const uint32_t* pred;
};

template <int NW>
struct Steps {
  const TablesW& tb;
  const TreeConsts& tc;
  Search<NW>& t;
  bool fresh;
  uint64_t reads = 0;

  void visit(const State<kTreeSlots>& s, Digits dg, uint32_t d) {
    if (d == tc.leaf_level) {
      store_node(s, dg, t.node.data(), 1u, 0u);
      node_to_window<NW>(t.node.data(), 1u, 0u, tc.W0, t.tw.n, t.slot.data(), 1u);
      const CountedTables<NW> sd{{t.sdw.f, &reads}, t.sdw.recip, t.sdw.pred};
      const uint32_t ncomb = tc.alone_last ? tc.combos / tc.radix : tc.combos;
      LaneBest lb;
      for (uint32_t c = 0; c < ncomb; ++c) {
        if (fresh) lb = LaneBest{};
        leaf_combos<NW>(t.tw, sd, t.rtw.data(), tc, t.slot.data(), 1u, dg, true, c, c + 1u, lb);
      }
      return;
    }
    for (uint32_t a = 0; a < tc.radix; ++a) {
      State<kTreeSlots> c = s;
      Digits cd = dg;
      if (expand_child<kTreeSlots>(tb, t.sd, t.rt.data(), tc, c, cd, d, a, kInfeasible, t.ef.data(), 1u))
        visit(c, cd, d + 1);
    }
  }
};
}  // namespace

extern "C" uint64_t host_unpruned_steps(const bf_scenario_desc* d, uint32_t space, int fresh) {
  TablesW t0, tb;
  host::build_tables(d, &t0);
  host::relabel_sources_first(t0, &tb);
  TreeConsts tc;
  host::tree_consts(tb, space, false, &tc);
  Search<32> search(tb, tc, kInfeasible);
  Steps<32> steps{tb, tc, search, fresh != 0};
  State<kTreeSlots> s;
  init_state(s, tb.all_mask);
  steps.visit(s, Digits{0u, 0u}, 0u);
  return steps.reads;
}

// The leaf modes of every leaf node that the expansions keep from `bound`:
// node_leaf_modes' sets, with the combinations leaf_mode_digits draws from them,
// against a simulation of all radix^D combinations of the node.  Returns how
// often a combination was listed twice or outside the sets, a list had another
// length than the product of the sets' sizes, or a combination with a makespan
// within the bound was not listed; *listed and *all count combinations.
namespace {
struct ModeCheck {
  const TablesW& tb;
  const TreeConsts& tc;
  Search<32>& t;
  uint32_t bound;
  uint64_t wrong = 0, listed = 0, all = 0;

  void leaf(const State<kTreeSlots>& s, Digits dg) {
    store_node(s, dg, t.node.data(), 1u, 0u);
    const uint32_t ncomb = tc.alone_last ? tc.combos / tc.radix : tc.combos, L = tc.leaf_level;
    std::vector<uint8_t> list(ncomb, 0);
    LeafModes modes;
    if (node_leaf_modes(t.node.data(), 1u, 0u, tb, tc, dg, bound, t.slot.data(), 1u, &modes)) {
      uint32_t product = 1;
      for (uint32_t v = 0; v < leaf_tools(tc); ++v) {
        const uint32_t b = 1u << (L + v);
        product *= ((modes.cpu & b) ? 1u : 0u) + ((modes.now & b) ? 1u : 0u) + ((modes.que & b) ? 1u : 0u);
      }
      const uint32_t combos = leaf_mode_combos(modes, tc);
      wrong += combos != product;
      listed += combos;
      for (uint32_t k = 0; k < combos; ++k) {
        const Digits d = leaf_mode_digits(modes, tc, k);
        uint32_t c = 0, place = 1;
        for (uint32_t v = 0; v < leaf_tools(tc); ++v, place *= tc.radix) {
          const uint32_t a = ((d.now >> v) & 1u) + 2u * ((d.que >> v) & 1u), b = 1u << (L + v);
          wrong += a > 2u || !((a == 0u ? modes.cpu : a == 1u ? modes.now : modes.que) & b);
          c += a * place;
        }
        wrong += c >= ncomb || list[c < ncomb ? c : 0]++ != 0;
      }
    }
    all += ncomb;
    node_to_window<32>(t.node.data(), 1u, 0u, tc.W0, t.tw.n, t.slot.data(), 1u);
    for (uint32_t c = 0; c < ncomb; ++c) {
      LaneBest lb;
      leaf_run<32, false>(t.tw, t.sdw, t.rtw.data(), tc, t.slot.data(), 1u, dg, leaf_digits(c, tc.radix, leaf_tools(tc), 0u), lb,
                   kInfeasible);
      wrong += lb.ms != kInfeasible && lb.ms <= bound && !list[c];
    }
  }

  void visit(const State<kTreeSlots>& s, Digits dg, uint32_t d) {
    if (d == tc.leaf_level) {
      leaf(s, dg);
      return;
    }
    for (uint32_t a = 0; a < tc.radix; ++a) {
      State<kTreeSlots> c = s;
      Digits cd = dg;
      if (expand_child<kTreeSlots>(tb, t.sd, t.rt.data(), tc, c, cd, d, a, bound, t.ef.data(), 1u)) visit(c, cd, d + 1);
    }
  }
};
}  // namespace

extern "C" uint64_t host_leaf_modes(const bf_scenario_desc* d, uint32_t space, uint32_t bound, uint64_t* listed,
                                    uint64_t* all) {
  TablesW t0, tb;
  host::build_tables(d, &t0);
  host::relabel_sources_first(t0, &tb);
  TreeConsts tc;
  host::tree_consts(tb, space, true, &tc);
  Search<32> search(tb, tc, bound);
  ModeCheck check{tb, tc, search, bound};
  State<kTreeSlots> s;
  init_state(s, tb.all_mask);
  check.visit(s, Digits{0u, 0u}, 0u);
  *listed = check.listed;
  *all = check.all;
  return check.wrong;
}
