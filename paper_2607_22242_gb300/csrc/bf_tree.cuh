// bf_tree.cuh -- the tree search: exact branch and bound over mode prefixes,
// for scenarios of up to 32 tools, over the full decision space (3 modes per
// tool) or the binary cpu/gpu_now space (§4.1: S1-S10 choose between CPU and
// GPU only).
//
// Tools are numbered as in the tables the search runs on (the scenario's
// tools with the sources first, host::relabel_sources_first); results carry
// canonical indices (TreeConsts::pow3).
//
// A node at level d assigns modes to tools [0, d) and holds the simulation
// state at its checkpoint: the first instant at which a tool >= d would
// become ready (bf_sim.cuh, resumable runs).  Until then no tool >= d has
// started, so that state is shared by every mapping extending the node.  A
// child assigns tool d and resumes the parent's state up to its own
// checkpoint.  Nodes at the leaf level L = n - D are not expanded further:
// the leaf kernel resumes each one for all radix^D modes of the last D tools
// and simulates them to the end.
//
// Pruning (Plan::bound's rule, with a per-node bound): the makespan of every
// mapping extending a node is at least the node's lower bound (below); a node
// whose bound exceeds the best makespan found so far (strictly) is dropped.
// The optimum and all its ties have every prefix within the bound, so the
// search returns the same (makespan, lowest index) as full enumeration.
#pragma once

#include "bf_plan.h"
#include "bf_sim.cuh"

namespace bfk {

constexpr int kTreeSlots = 32;
using TablesW = TablesT<kTreeSlots>;
using SmemTablesW = SmemTablesT<kTreeSlots>;

// Leaf window widths compiled for the leaf kernel: a window of nw tools runs
// in the narrowest that holds it.
#define BF_TREE_BUCKETS(X) X(8) X(12) X(16) X(20) X(24) X(32)

// Per-scenario constants of a tree search.
struct TreeConsts {
  uint32_t n;
  uint32_t radix;        // 2: {cpu, gpu_now}; 3: {cpu, gpu_now, gpu_queue}
  uint32_t leaf_level;   // L: nodes at this level go to the leaf kernel
  uint32_t D;            // n - L tools enumerated per leaf node
  uint32_t combos;       // radix^D
  uint32_t prune;        // 0: keep every node (full enumeration)
  uint32_t W0;           // leaf window start: tools below it have ended at every leaf checkpoint
  // 1 when every other tool precedes the last one: when it becomes ready it
  // runs alone, and ends alone[a] after that instant in mode a (0xFFFFFFFF: a
  // GPU mode over budget) -- the model's one remaining event at k = 1.
  uint32_t alone_last;
  uint32_t alone[3];
  uint32_t dmin[kTreeSlots];   // min(c, g + x): no mode runs tool v faster
  uint32_t sdown[kTreeSlots];  // longest path in dmin through v's successors (0 for a sink)
  // 1 when the tools are renumbered (sources first): tree slot v holds tool
  // orig[v] of the scenario, and ties compare canonical indices.
  uint32_t relabeled;
  uint64_t pow3[kTreeSlots];   // 3^(scenario position) of each slot's tool
  // pow3 when ties need it (renumbered tools), else nullptr.
  __device__ __forceinline__ const uint64_t* tie_pow3() const { return relabeled ? pow3 : nullptr; }
};

// A saved node: the state's words, then the digit masks; [word][node] layout
// with stride `cap` (nodes of one level sit side by side, so a warp's accesses
// to one word coalesce).
template <int NT>
struct NodeWords {
  static constexpr int value = 2 * NT + 11;
};

template <int NT>
__device__ __forceinline__ void store_node(const State<NT>& s, Digits dg, uint32_t* buf, uint32_t cap, uint32_t j) {
  uint32_t* p = buf + j;
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    p[(size_t)(2 * i) * cap] = s.ec[i];
    p[(size_t)(2 * i + 1) * cap] = s.eg[i];
  }
  p += (size_t)(2 * NT) * cap;
  p[0 * (size_t)cap] = s.done;
  p[1 * (size_t)cap] = s.pend;
  p[2 * (size_t)cap] = s.run_g;
  p[3 * (size_t)cap] = s.qwait;
  p[4 * (size_t)cap] = s.T;
  p[5 * (size_t)cap] = s.V;
  p[6 * (size_t)cap] = s.L;
  p[7 * (size_t)cap] = s.tc;
  p[8 * (size_t)cap] = s.gmin;
  p[9 * (size_t)cap] = dg.now;
  p[10 * (size_t)cap] = dg.que;
}

template <int NT>
__device__ __forceinline__ void load_node(const uint32_t* buf, uint32_t cap, uint32_t j, State<NT>& s, Digits& dg) {
  const uint32_t* p = buf + j;
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    s.ec[i] = p[(size_t)(2 * i) * cap];
    s.eg[i] = p[(size_t)(2 * i + 1) * cap];
  }
  p += (size_t)(2 * NT) * cap;
  s.done = p[0 * (size_t)cap];
  s.pend = p[1 * (size_t)cap];
  s.run_g = p[2 * (size_t)cap];
  s.qwait = p[3 * (size_t)cap];
  s.T = p[4 * (size_t)cap];
  s.V = p[5 * (size_t)cap];
  s.L = p[6 * (size_t)cap];
  s.tc = p[7 * (size_t)cap];
  s.gmin = p[8 * (size_t)cap];
  dg.now = p[9 * (size_t)cap];
  dg.que = p[10 * (size_t)cap];
}

// Per-slot end times of a node saved in HBM.
struct NodeSlots {
  const uint32_t* p;  // word 0 of the node
  uint32_t cap;
  __device__ __forceinline__ uint32_t ec(int v) const { return p[(size_t)(2 * v) * cap]; }
  __device__ __forceinline__ uint32_t eg(int v) const { return p[(size_t)(2 * v + 1) * cap]; }
};

// Copy node j of a level buffer into a lane's shared-memory state over the
// window [W0, W0 + NW) (slots past the last tool: no CPU end, stamp 0), with
// masks shifted to window numbering.  Every tool below W0 has ended at every
// leaf node's checkpoint, and no running tool lies outside the window.
template <int NW>
__device__ __forceinline__ void node_to_window(const uint32_t* buf, uint32_t cap, uint32_t j, uint32_t W0,
                                               uint32_t nw, uint32_t* slot, uint32_t stride) {
  const uint32_t* p = buf + j;
#pragma unroll
  for (int i = 0; i < NW; ++i) {
    const uint32_t v = W0 + (uint32_t)i;
    const bool in = v < (uint32_t)kTreeSlots;
    slot[(2 * i) * stride] = in ? p[(size_t)(2 * v) * cap] : 0xFFFFFFFFu;
    slot[(2 * i + 1) * stride] = in ? p[(size_t)(2 * v + 1) * cap] : 0u;
  }
  const uint32_t* t = p + (size_t)(2 * kTreeSlots) * cap;
  const uint32_t wmask = nw >= 32u ? 0xFFFFFFFFu : ((1u << nw) - 1u);
  uint32_t* q = slot + (2 * NW) * stride;
  q[0 * stride] = (t[0 * (size_t)cap] >> W0) | ~wmask;  // done
  q[1 * stride] = (t[1 * (size_t)cap] >> W0) & wmask;   // pend
  q[2 * stride] = t[2 * (size_t)cap] >> W0;             // run_g
  q[3 * stride] = t[3 * (size_t)cap] >> W0;             // qwait
  q[4 * stride] = t[4 * (size_t)cap];                   // T
  q[5 * stride] = t[5 * (size_t)cap];                   // V
  q[6 * stride] = t[6 * (size_t)cap];                   // L
  q[7 * stride] = t[7 * (size_t)cap];                   // tc
  q[8 * stride] = t[8 * (size_t)cap];                   // gmin
}

// Lower bound on the makespan of every mapping that extends a node whose state
// `s` is at a checkpoint (before the admission at s.T), with the modes of the
// tools in `known` given by `dg`.  The earliest finish EF of every unfinished
// tool, in index (topological) order, is
//   * a running CPU tool's end time (exact);
//   * T + ceil(r / 1024) of a running GPU tool with r work units left: f[k] >=
//     f[1] = 1024, and the model rounds GPU progress down and completion times up;
//   * of any other tool the latest of T and its unfinished predecessors' EF, plus
//     its duration in its mode (c, g + x or l + g + x; min(c, g + x) if open).
// No tool starts before T or before its predecessors end, so EF never exceeds
// the true end, and the makespan is at least the largest EF.  Queued tools run
// one at a time, so it is also at least T + the sum of the remaining durations of
// the unfinished tools known to be queued.  `ef` is a per-thread column of NT
// words in shared memory (stride `stride`).  Times fit in 32 bits: T plus the
// durations of a chain of remaining tools stays below the validated makespan
// bound.
template <int NT, typename TB>
__device__ __forceinline__ uint32_t forward_bound(const State<NT>& s, const TB& tb, const TreeConsts& tc, Digits dg,
                                                  uint32_t known, uint32_t* ef, uint32_t stride) {
  const uint32_t T = s.T;
  uint32_t lb = T, qsum = 0u;
#pragma unroll
  for (int v = 0; v < NT; ++v) {
    const uint32_t bit = 1u << v;
    if (s.done & bit) continue;
    uint32_t fin;
    if (s.ec[v] != 0xFFFFFFFFu) {
      fin = s.ec[v];
    } else if (s.run_g & bit) {
      const uint32_t r = s.eg[v] - s.V;
      const uint32_t left = (r >> 10) + ((r & 1023u) != 0u);
      fin = T + left;
      if (dg.que & bit) qsum += left;
    } else {
      uint32_t d = tc.dmin[v];
      if (known & bit) {
        d = (dg.now & bit) ? (tb.wnow[v] >> 10) : (dg.que & bit) ? (tb.wq[v] >> 10) : tb.cpu[v];
        if (dg.que & bit) qsum += d;
      }
      uint32_t start = T;
      for (uint32_t m = tb.pred[v] & ~s.done; m; m &= m - 1u) start = max(start, ef[(__ffs(m) - 1) * stride]);
      fin = start + d;
    }
    ef[v * stride] = fin;
    lb = max(lb, fin);
  }
  return max(lb, T + qsum);
}

// Child (tool d in mode a) of the node whose state and digits are in s / dg,
// advanced in place to the child's checkpoint.  Returns false when every
// mapping below the child is infeasible or, with pruning, provably worse
// than `bound` (forward_bound, scratch column `ef`).  Requires d + 1 < n.
template <int NT, typename TB, typename SD>
__device__ __forceinline__ bool expand_child(const TB& tb, const SD& sd, const uint32_t* rt, const TreeConsts& tc,
                                             State<NT>& s, Digits& dg, uint32_t d, uint32_t a, uint32_t bound,
                                             uint32_t* ef, uint32_t stride) {
  const uint32_t bit = 1u << d;
  if (a == 1u) dg.now |= bit;
  if (a == 2u) {
    if (tb.big_mask & bit) return false;  // a queued tool with m > M never starts
    dg.que |= bit;
  }
  const uint32_t assigned = (bit << 1) - 1u;  // tools [0, d]; all ones for d = 31
  if (run<NT>(s, tb, sd, rt, dg, tb.all_mask & ~assigned) != kRunStopped) return false;
  return !tc.prune || forward_bound<NT>(s, tb, tc, dg, assigned, ef, stride) <= bound;
}

// Node of the first d0 tools' modes `dg`, simulated from time 0 (s holds the
// initial state): expand_child's test for d0 tools at once.
template <int NT, typename TB, typename SD>
__device__ __forceinline__ bool expand_start(const TB& tb, const SD& sd, const uint32_t* rt, const TreeConsts& tc,
                                             State<NT>& s, Digits dg, uint32_t d0, uint32_t bound, uint32_t* ef,
                                             uint32_t stride) {
  if (dg.que & tb.big_mask) return false;
  const uint32_t assigned = (1u << d0) - 1u;
  if (run<NT>(s, tb, sd, rt, dg, tb.all_mask & ~assigned) != kRunStopped) return false;
  return !tc.prune || forward_bound<NT>(s, tb, tc, dg, assigned, ef, stride) <= bound;
}

// The modes that each leaf tool may take in a mapping no worse than the bound,
// as tool sets.
struct LeafModes {
  uint32_t cpu, now, que;
};

// The forward bound of leaf node j (forward_bound, over the leaf window, read
// word by word from HBM) with the leaf tools open: false when every mapping
// below the node is worse than `bound`; else *out has the modes of each leaf
// tool in which it can end, with the longest minimum path after it, within the
// bound (a GPU mode over the whole budget never starts).  A tool's earliest end
// is the least over the modes it keeps.  `ef`: a column of the window's width
// in shared memory.
template <typename TB>
__device__ __forceinline__ bool node_leaf_modes(const uint32_t* buf, uint32_t cap, uint32_t j, const TB& tb,
                                                const TreeConsts& tc, Digits dg, uint32_t bound, uint32_t* ef,
                                                uint32_t stride, LeafModes* out) {
  const NodeSlots slot{buf + j, cap};
  const uint32_t* t = buf + j + (size_t)(2 * kTreeSlots) * cap;
  const uint32_t done = t[0], run_g = t[2 * (size_t)cap], T = t[4 * (size_t)cap], V = t[5 * (size_t)cap];
  *out = LeafModes{0u, 0u, 0u};
  uint64_t qsum = 0u;
  for (uint32_t v = tc.W0; v < tc.n; ++v) {
    const uint32_t bit = 1u << v;
    if (done & bit) continue;
    const uint32_t ec = slot.ec((int)v);
    uint64_t fin = ~0ull;
    if (ec != 0xFFFFFFFFu) {
      fin = ec;
    } else if (run_g & bit) {
      const uint32_t r = slot.eg((int)v) - V;
      const uint32_t left = (r >> 10) + ((r & 1023u) != 0u);
      fin = (uint64_t)T + left;
      if (dg.que & bit) qsum += left;
    } else {
      uint64_t start = T;
      for (uint32_t m = tb.pred[v] & ~done; m; m &= m - 1u) {
        const uint32_t e = ef[(__ffs(m) - 1u - tc.W0) * stride];
        start = e > start ? e : start;
      }
      const uint32_t dc = tb.cpu[v], dn = tb.wnow[v] >> 10, dq = tb.wq[v] >> 10;
      if (v < tc.leaf_level) {
        fin = start + ((dg.now & bit) ? dn : (dg.que & bit) ? dq : dc);
        if (dg.que & bit) qsum += dq;
      } else {
        const uint64_t after = start + tc.sdown[v];
        const bool gpu = (tb.big_mask & bit) == 0u;
        if (after + dc <= bound) {
          out->cpu |= bit;
          fin = start + dc;
        }
        if (gpu && after + dn <= bound) {
          out->now |= bit;
          fin = start + dn < fin ? start + dn : fin;
        }
        if (gpu && tc.radix == 3u && after + dq <= bound) {
          out->que |= bit;
          fin = start + dq < fin ? start + dq : fin;
        }
        if (fin == ~0ull) return false;
      }
    }
    if (fin + tc.sdown[v] > bound) return false;
    ef[(v - tc.W0) * stride] = (uint32_t)fin;
  }
  return T + qsum <= bound;
}

// Digits of leaf combination c (tools [L, n)), as masks shifted to tool L.
__device__ __forceinline__ Digits leaf_digits(uint32_t c, uint32_t radix, uint32_t D, uint32_t L) {
  if (radix == 2u) return Digits{c << L, 0u};
  const Digits d = decode(c, D);
  return Digits{d.now << L, d.que << L};
}

// Canonical index of a mapping given as digit masks.
__device__ __forceinline__ uint64_t index_of(Digits dg, const uint64_t* pow3) {
  uint64_t idx = 0;
  for (uint32_t m = dg.now; m; m &= m - 1u) idx += pow3[__ffs(m) - 1];
  for (uint32_t m = dg.que; m; m &= m - 1u) idx += 2u * pow3[__ffs(m) - 1];
  return idx;
}

// a < b in slot order: the highest slot whose digits differ decides (the
// canonical order when the slots are not renumbered).
__device__ __forceinline__ bool index_less(Digits a, Digits b) {
  const uint32_t diff = (a.now ^ b.now) | (a.que ^ b.que);
  if (diff == 0u) return false;
  const uint32_t top = 1u << (31 - __clz(diff));
  const uint32_t da = ((a.now & top) ? 1u : 0u) + ((a.que & top) ? 2u : 0u);
  const uint32_t db = ((b.now & top) ? 1u : 0u) + ((b.que & top) ? 2u : 0u);
  return da < db;
}

// Best mapping seen: lowest makespan, ties to the lowest canonical index.
// pow3 (TreeConsts::tie_pow3) is nullptr when slot order is the scenario's
// order; otherwise ties compare the canonical indices it gives.
struct LaneBest {
  uint32_t ms = kInfeasible;
  Digits dg{0u, 0u};
  __device__ __forceinline__ void offer(uint32_t m, Digits d, const uint64_t* pow3) {
    if (m < ms ||
        (m == ms && m != kInfeasible && (pow3 ? index_of(d, pow3) < index_of(dg, pow3) : index_less(d, dg)))) {
      ms = m;
      dg = d;
    }
  }
};

// Simulate one combination `dc` of the leaf tools' modes (bit 0: tool L) of the
// leaf node saved in `slot` (a lane's shared-memory window state, stride
// `stride`) whose digits are `dg` (all tools); tw/sdw/rtw are the window's
// tables.  PRUNE: a run past `bound` or the best so far is given up; unpruned,
// every run goes to its end (compiled without the test: all 2^32 binary mappings
// of a 32-tool spine 115.7 -> 111.9 ms).  False when the combination was not
// simulated (a queued tool larger than the budget).
// With tc.alone_last, dc are modes of the leaf tools but the last one: the run
// goes on until the last tool becomes ready (everything else has ended then)
// and yields one makespan per mode of the last tool.
template <int NW, bool PRUNE, typename TBW, typename SD>
__device__ __forceinline__ bool leaf_run(const TBW& tw, const SD& sdw, const uint32_t* rtw, const TreeConsts& tc,
                                         const uint32_t* slot, uint32_t stride, Digits dg, Digits dc, LaneBest& best,
                                         uint32_t bound) {
  const uint32_t L = tc.leaf_level, W0 = tc.W0, last = tc.n - 1u, lastw = last - W0;
  const Digits full{dg.now | (dc.now << L), dg.que | (dc.que << L)};
  const Digits sim{full.now >> W0, full.que >> W0};
  if (sim.que & tw.big_mask) return false;
  State<NW> w;
  load_lane(slot, stride, w);
  const uint32_t limit = !PRUNE ? kInfeasible : best.ms < bound ? best.ms : bound;
  if (tc.alone_last) {
    if (run<NW>(w, tw, sdw, rtw, sim, 1u << lastw, 1u << lastw, limit) != kRunStopped) return true;  // infeasible before it
    for (uint32_t a = 0; a < tc.radix; ++a) {
      if (tc.alone[a] == kInfeasible) continue;
      best.offer(w.T + tc.alone[a],
                 Digits{full.now | (a == 1u ? 1u << last : 0u), full.que | (a == 2u ? 1u << last : 0u)},
                 tc.tie_pow3());
    }
  } else if (run<NW>(w, tw, sdw, rtw, sim, 0u, 0u, limit) == kRunFinished) {
    best.offer(w.T, full, tc.tie_pow3());
  }
  return true;
}

// Leaf tools whose modes a leaf run enumerates (all but a lone last one).
__device__ __forceinline__ uint32_t leaf_tools(const TreeConsts& tc) { return tc.alone_last ? tc.D - 1u : tc.D; }

// Combinations [c0, c1) of a leaf node's modes (leaf_run), all of them; returns
// how many were simulated.  `valid` false runs the loop without work (lanes of a
// warp stay in lockstep).
template <int NW, typename TBW, typename SD>
__device__ __forceinline__ uint32_t leaf_combos(const TBW& tw, const SD& sdw, const uint32_t* rtw,
                                                const TreeConsts& tc, const uint32_t* slot, uint32_t stride, Digits dg,
                                                bool valid, uint32_t c0, uint32_t c1, LaneBest& best) {
  uint32_t ran = 0u;
  for (uint32_t c = c0; c < c1; ++c) {
    if (!valid) continue;
    ran += leaf_run<NW, false>(tw, sdw, rtw, tc, slot, stride, dg, leaf_digits(c, tc.radix, leaf_tools(tc), 0u), best,
                               kInfeasible) ? 1u : 0u;
  }
  return ran;
}

// Combinations of the leaf tools' modes that `modes` leaves (0 if a tool has
// none), and the k-th of them: a mixed-radix number, the first leaf tool least
// significant, each digit counting the modes its tool keeps.
__device__ __forceinline__ uint32_t leaf_mode_combos(const LeafModes& modes, const TreeConsts& tc) {
  uint32_t count = 1u;
  for (uint32_t t = 0; t < leaf_tools(tc); ++t) {
    const uint32_t bit = 1u << (tc.leaf_level + t);
    count *= ((modes.cpu & bit) ? 1u : 0u) + ((modes.now & bit) ? 1u : 0u) + ((modes.que & bit) ? 1u : 0u);
  }
  return count;
}

__device__ __forceinline__ Digits leaf_mode_digits(const LeafModes& modes, const TreeConsts& tc, uint32_t k) {
  Digits d{0u, 0u};
  for (uint32_t t = 0; t < leaf_tools(tc); ++t) {
    const uint32_t bit = 1u << (tc.leaf_level + t);
    const bool c = modes.cpu & bit, n = modes.now & bit, q = modes.que & bit;
    const uint32_t r = (c ? 1u : 0u) + (n ? 1u : 0u) + (q ? 1u : 0u);
    const uint32_t next = r == 3u ? k / 3u : (r == 2u ? k >> 1 : k), j = k - next * r;
    k = r == 1u ? k : next;
    const uint32_t at = r == 1u ? 0u : j;  // the at-th mode the tool keeps
    const uint32_t mode = at == 0u ? (c ? 0u : (n ? 1u : 2u)) : (at == 1u ? (c && n ? 1u : 2u) : 2u);
    d.now |= mode == 1u ? 1u << t : 0u;
    d.que |= mode == 2u ? 1u << t : 0u;
  }
  return d;
}

// The makespans a search prunes by, in device memory.  `live` is the best one
// known; the blocks of a leaf launch lower it while others of the same launch
// start.  `leaf` is what `live` was before the coming leaf launch (the start and
// expansion kernels copy it, and only leaf launches change `live`): the tasks
// of a node group cut one list of combinations into parts, so that list must be
// the same for all of them.
struct TreeBounds {
  uint32_t live, leaf;
};

__device__ __forceinline__ uint32_t read_bound(const uint32_t* bound) {
  return *reinterpret_cast<const volatile uint32_t*>(bound);
}

// A warp task of the leaf kernel: part `part` of `parts` of the mappings below
// the 32 nodes of group `g`, one node's modes and state prepared by each lane.
// Unpruned, the lanes walk the combinations [part * chunk, (part + 1) * chunk) of
// their own nodes in lockstep, which keeps them on one path (99 %).  Pruned, the
// combinations that the bound leaves differ from node to node (a handful of 243
// in some, none in most): while the nodes keep about as many each, every lane
// walks its own node's; else (fewer than 12 times the fullest node's in all) they
// are dealt to the lanes one by one over all 32 nodes, a lane resuming the state
// of whichever node its combination belongs to (and leaving the others' path).
// Own nodes only / dealt only / by this rule: full searches of 14 layered tools
// 0.29 / 0.30 / 0.28 ms, 20 tools 0.73 / 0.81 / 0.76, binary space of 24 tools 0.56
// / 0.70 / 0.59, geometric mean of 24 searches of 8 to 26 tools 0.29 / 0.37 / 0.29;
// searches with millions of leaf nodes, which keep the whole grid busy, gain by
// dealing more often than the rule does: 28 tools in 16 GiB 382 / 175 / 420 ms, 32
// tools 187 / 131 / 230.
// Modes, totals and that choice depend on the nodes and on bounds->leaf alone, so
// that the parts of a group are parts of one list whenever they run; the live
// bound only gives up single runs.
// `slot`: this lane's window state in shared memory (stride STRIDE, the warp's 32
// lanes side by side).  Every lane of the warp calls it.  Returns the
// combinations this lane simulated; *nodes has the lanes with a node to enumerate.
template <int NW, uint32_t STRIDE, typename TB, typename TBW, typename SD>
__device__ __forceinline__ uint32_t leaf_task(const TB& tb, const TBW& tw, const SD& sdw, const uint32_t* rtw,
                                              const TreeConsts& tc, const uint32_t* buf, uint32_t cap, uint32_t cnt,
                                              uint32_t g, uint32_t part, uint32_t parts, uint32_t chunk,
                                              const TreeBounds* bounds, uint32_t* slot, LaneBest& best,
                                              uint32_t* nodes) {
  const uint32_t lane = threadIdx.x & 31u, j = g * 32u + lane;
  bool valid = j < cnt;
  Digits dg{0u, 0u};
  LeafModes modes{0u, 0u, 0u};
  const uint32_t kept = tc.prune ? read_bound(&bounds->leaf) : kInfeasible;
  uint32_t limit = kept;  // of single runs: falls with the live bound
  __syncwarp();  // the other lanes are done with this lane's state
  if (valid) {
    const uint32_t* t = buf + j + (size_t)(2 * kTreeSlots) * cap;
    dg = Digits{t[9 * (size_t)cap], t[10 * (size_t)cap]};
    // The incumbent may have improved since this node was bounded; only modes
    // within it are enumerated.
    if (tc.prune) valid = node_leaf_modes(buf, cap, j, tb, tc, dg, kept, slot, STRIDE, &modes);
    if (valid) node_to_window<NW>(buf, cap, j, tc.W0, tw.n, slot, STRIDE);
  }
  __syncwarp();  // dealt combinations resume other lanes' states: votes and shuffles order no memory
  *nodes = __ballot_sync(0xFFFFFFFFu, valid);
  if (*nodes == 0u) return 0u;
  uint32_t ran = 0u;
  uint32_t upto = valid && tc.prune ? leaf_mode_combos(modes, tc) : 0u;  // combinations of lanes 0 .. this one
  const uint32_t most = __reduce_max_sync(0xFFFFFFFFu, upto), sum = __reduce_add_sync(0xFFFFFFFFu, upto);
  if (tc.prune && sum < most * 12u) {
#pragma unroll
    for (uint32_t o = 1; o < 32u; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, upto, o);
      if (lane >= o) upto += v;
    }
    const uint32_t total = __shfl_sync(0xFFFFFFFFu, upto, 31);
    const uint32_t q0 = (uint32_t)((uint64_t)total * part / parts), q1 = (uint32_t)((uint64_t)total * (part + 1u) / parts);
    for (uint32_t base = q0; base < q1; base += 32u) {
      const uint32_t q = min(base + lane, q1 - 1u);
      uint32_t i = 0u;  // the node whose combinations include the q-th: the first lane with upto > q
#pragma unroll
      for (uint32_t step = 16; step; step >>= 1)
        if (__shfl_sync(0xFFFFFFFFu, upto, i + step - 1u) <= q) i += step;
      const uint32_t before = __shfl_sync(0xFFFFFFFFu, upto, i ? i - 1u : 0u);
      const LeafModes m{__shfl_sync(0xFFFFFFFFu, modes.cpu, i), __shfl_sync(0xFFFFFFFFu, modes.now, i),
                        __shfl_sync(0xFFFFFFFFu, modes.que, i)};
      const Digits d{__shfl_sync(0xFFFFFFFFu, dg.now, i), __shfl_sync(0xFFFFFFFFu, dg.que, i)};
      if (base + lane < q1) {
        limit = min(limit, read_bound(&bounds->live));
        const Digits dc = leaf_mode_digits(m, tc, q - (i ? before : 0u));
        ran += leaf_run<NW, true>(tw, sdw, rtw, tc, slot + (int)(i - lane), STRIDE, d, dc, best, limit) ? 1u : 0u;
      }
      __syncwarp();
    }
  } else if (tc.prune) {
    const uint32_t q0 = upto * part / parts, q1 = upto * (part + 1u) / parts;
    const uint32_t rounds = __reduce_max_sync(0xFFFFFFFFu, q1 - q0);
    for (uint32_t k = 0; k < rounds; ++k) {
      if (q0 + k < q1) {
        limit = min(limit, read_bound(&bounds->live));
        ran += leaf_run<NW, true>(tw, sdw, rtw, tc, slot, STRIDE, dg, leaf_mode_digits(modes, tc, q0 + k), best, limit) ? 1u : 0u;
      }
      __syncwarp();
    }
  } else {
    const uint32_t c0 = part * chunk, c1 = min(c0 + chunk, tc.alone_last ? tc.combos / tc.radix : tc.combos);
    ran = leaf_combos<NW>(tw, sdw, rtw, tc, slot, STRIDE, dg, valid, c0, c1, best);
  }
  return ran;
}

namespace host {

// Constants of a search over tables tb (the scenario's tools, renumbered or
// not) in the space of radix R (2: binary, 3: full): the leaf depth D (5 tools
// in the full space, 8 in the binary one, all of them for smaller scenarios),
// the leaf window, the lone last tool's durations, the per-tool minimum
// durations and downstream paths of the bounds, and each slot's place value
// in the canonical index.
inline void tree_consts(const TablesW& tb, uint32_t R, bool prune, TreeConsts* out) {
  TreeConsts& tc = *out;
  std::memset(&tc, 0, sizeof tc);
  const uint32_t n = tb.n;
  tc.n = n;
  tc.radix = R;
  tc.D = n < (R == 3 ? 5u : 8u) ? n : (R == 3 ? 5u : 8u);
  tc.leaf_level = n - tc.D;
  tc.combos = 1;
  for (uint32_t i = 0; i < tc.D; ++i) tc.combos *= R;
  tc.prune = prune ? 1u : 0u;
  tc.W0 = window_start(tb, tc.leaf_level);
  {
    uint32_t anc[kTreeSlots];
    ancestors(tb, anc);
    const uint32_t last = n - 1, others = (last >= 32u) ? ~0u : ((1u << last) - 1u);
    tc.alone_last = (tc.D >= 1u && (anc[last] & others) == others) ? 1u : 0u;
    const bool fits = tb.vram[last] <= tb.budget;
    tc.alone[0] = tb.cpu[last];
    tc.alone[1] = fits ? tb.wnow[last] >> 10 : 0xFFFFFFFFu;
    tc.alone[2] = fits ? tb.wq[last] >> 10 : 0xFFFFFFFFu;
  }
  uint64_t down[kTreeSlots] = {0};
  for (int v = (int)n - 1; v >= 0; --v) {
    const uint32_t gpu = tb.wnow[v] >> 10;
    tc.dmin[v] = tb.cpu[v] < gpu ? tb.cpu[v] : gpu;
    uint64_t longest = 0;
    for (uint32_t w = (uint32_t)v + 1; w < n; ++w)
      if ((tb.succ[v] >> w) & 1u) longest = down[w] > longest ? down[w] : longest;
    tc.sdown[v] = (uint32_t)(longest < 0xFFFFFFFFull ? longest : 0xFFFFFFFFull);
    down[v] = tc.dmin[v] + longest;
  }
  for (uint32_t i = 0; i < (uint32_t)kTreeSlots; ++i) tc.pow3[i] = pow3(i < n ? tb.orig[i] : i);
  tc.relabeled = tb.relabeled ? 1u : 0u;
}

}  // namespace host
}  // namespace bfk
