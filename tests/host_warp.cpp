// Host build of device code whose lanes work together (tests/host_warp.h), for
// tests that run without a GPU.  Test infrastructure only.
#include <algorithm>
#include <cstdint>
#include <cstring>
#include <vector>

#define BF_HOST_WARP
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

#include "../paper_2607_22242_gb300/csrc/bf_plan.h"
#include "../paper_2607_22242_gb300/csrc/bf_tree.cuh"

using namespace bfk;

// The lane-tree search of one scenario by one warp with levels [0, x), [x, y),
// [y, n), lanes without a root taking over part of another's work
// (lt_lane<SHARE>).  Every mapping reported is stored at its canonical index;
// out[] starts at 0xFFFFFFFF, a second report of one index stores 0xDEADBEEF.
// *shared: how often a lane went on after it had found no root.
template <uint32_t NC, uint32_t W>
static int lanetree_warp(const bf_scenario_desc* d, uint32_t x, uint32_t y, uint32_t* out, uint32_t* shared) {
  LaneTreeRecord rec;
  host::lanetree_record(d, &rec);
  rec.x = x;
  rec.y = y;
  const uint64_t total = host::pow3(d->n);
  for (uint64_t j = 0; j < total; ++j) out[j] = 0xFFFFFFFFu;
  std::vector<LtSharedT<NC>> tables(1);
  LtSharedT<NC>& S = tables[0];
  S.rec = rec;
  threadIdx.x = 0;
  blockDim.x = 1;
  lt_fill_tables(S);
  struct Store {
    uint32_t* out;
    bool* rootless;
    uint32_t* shared;
    void operator()(uint32_t idx, uint32_t ms) {
      out[idx] = out[idx] == 0xFFFFFFFFu ? ms : 0xDEADBEEFu;
      *shared += *rootless ? 1u : 0u;
    }
  };
  const uint32_t roots = (uint32_t)host::pow3(x);
  uint32_t next = 0;
  *shared = 0;
  const std::vector<uint32_t> stale((size_t)lt_rows<W>(d->n) * hostwarp::kLanes, 0xA5A5A5A5u);
  return hostwarp::run(stale, [&](unsigned lane) {
    bool rootless = false;
    Store sink{out, &rootless, shared};
    lt_lane<NC, W, false, false, true>(S, hostwarp::shared() + lane, hostwarp::kLanes,
                                       [&]() {
                                         rootless = next >= roots;
                                         return rootless ? 0xFFFFFFFFu : next++;
                                       },
                                       sink);
  });
}

extern "C" int host_lanetree_warp(const bf_scenario_desc* d, uint32_t x, uint32_t y, int wide, uint32_t* out,
                                  uint32_t* shared) {
  if (x < 1 || x > y || y > d->n || y - x > kLtPartTools || d->n - y > kLtPartTools) return -1;
  return wide ? lanetree_warp<4, 1>(d, x, y, out, shared) : lanetree_warp<2, 0>(d, x, y, out, shared);
}

namespace {

// The leaf level of a tree search over the space of radix `space`: every node
// whose expansions survive `bound`, saved as the kernels save them.
struct LeafLevel {
  TablesW tb;
  TreeConsts tc;
  std::vector<uint32_t> nodes;  // [word][node]
  uint32_t cap = 0, count = 0;

  LeafLevel(const bf_scenario_desc* d, uint32_t space, bool prune, uint32_t bound) {
    TablesW t0;
    host::build_tables(d, &t0);
    host::relabel_sources_first(t0, &tb);
    host::tree_consts(tb, space, prune, &tc);
    SmemTablesW sd;
    std::vector<uint32_t> rt(ReadyTable<kTreeSlots>::size), ef(kTreeSlots);
    load_smem_tables(tb, sd);
    fill_ready_table<kTreeSlots>(tb, rt.data());
    std::vector<std::pair<State<kTreeSlots>, Digits>> level(1), next;
    init_state(level[0].first, tb.all_mask);
    level[0].second = Digits{0u, 0u};
    for (uint32_t dep = 0; dep < tc.leaf_level; ++dep, level.swap(next)) {
      next.clear();
      for (const auto& node : level)
        for (uint32_t a = 0; a < tc.radix; ++a) {
          auto c = node;
          if (expand_child<kTreeSlots>(tb, sd, rt.data(), tc, c.first, c.second, dep, a, bound, ef.data(), 1u))
            next.push_back(c);
        }
    }
    cap = count = (uint32_t)level.size();
    nodes.resize((size_t)NodeWords<kTreeSlots>::value * cap + 1u);
    for (uint32_t j = 0; j < count; ++j) store_node(level[j].first, level[j].second, nodes.data(), cap, j);
  }
};

template <int NW>
int leaf_warps(const LeafLevel& L, uint32_t start, uint32_t parts, const uint32_t* bounds, uint64_t* out) {
  const TreeConsts& tc = L.tc;
  TablesT<NW> tw;
  host::build_window(L.tb, tc.W0, &tw);
  SmemTablesT<NW> sdw;
  std::vector<uint32_t> rtw(ReadyTable<NW>::size);
  load_smem_tables(tw, sdw);
  fill_ready_table<NW>(tw, rtw.data());
  const uint32_t ncomb = tc.alone_last ? tc.combos / tc.radix : tc.combos;
  const std::vector<uint32_t> stale((size_t)LaneWords<NW>::value * hostwarp::kLanes, 0xA5A5A5A5u);
  uint64_t ms = ~0ull, idx = ~0ull, ran = 0, nodes = 0;
  for (uint32_t g = 0; g < (L.count + 31u) / 32u; ++g)
    for (uint32_t part = 0; part < parts; ++part) {
      const TreeBounds bound{bounds[part], start};
      const int err = hostwarp::run(stale, [&](unsigned lane) {
        LaneBest best;
        uint32_t live;
        ran += leaf_task<NW, hostwarp::kLanes>(L.tb, tw, sdw, rtw.data(), tc, L.nodes.data(), L.cap, L.count, g, part,
                                               parts, (ncomb + parts - 1u) / parts, &bound, hostwarp::shared() + lane,
                                               best, &live);
        if (part == 0 && lane == 0) nodes += (uint64_t)__popc(live);
        if (best.ms == kInfeasible) return;
        const uint64_t i = index_of(best.dg, tc.pow3);
        if (best.ms < ms || (best.ms == ms && i < idx)) {
          ms = best.ms;
          idx = i;
        }
      });
      if (err) return err;
    }
  out[0] = ms;
  out[1] = idx;
  out[2] = ran * (tc.alone_last ? tc.radix : 1u);
  out[3] = nodes;
  out[4] = L.count;
  return 0;
}

}  // namespace

// The leaf kernel's tasks over every leaf node that the expansions keep from
// `start`, which is also the leaf launch's bound, `parts` tasks per group of 32
// nodes, task p with the live bound at bounds[p].  out[0..4] = best makespan (~0: none), its canonical index,
// mappings simulated, nodes enumerated by the groups' first tasks, leaf nodes.
extern "C" int host_leaf_warps(const bf_scenario_desc* d, uint32_t space, int prune, uint32_t start, uint32_t parts,
                               const uint32_t* bounds, uint64_t* out) {
  threadIdx.x = 0;
  blockDim.x = 1;
  const LeafLevel L(d, space, prune != 0, start);
  const uint32_t nw = L.tb.n - L.tc.W0;
#define BF_TRY(NW) \
  if (nw <= (uint32_t)NW) return leaf_warps<NW>(L, start, parts, bounds, out);
  BF_TREE_BUCKETS(BF_TRY)
#undef BF_TRY
  return -1;
}
