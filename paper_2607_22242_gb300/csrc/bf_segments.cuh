// bf_segments.cuh -- evaluations, and searches by branch and bound, of
// scenarios whose DAG has barriers: the plan, its host side and the sum of a
// mapping's table entries (kernels in bf_segments.cu).
//
// A barrier at c is a place in the numbering where every tool >= c has every
// tool < c among its ancestors.  The instant the first tool >= c becomes
// ready, all tools below c have ended: nothing runs, nothing waits, no VRAM
// is held, and the model's arithmetic depends only on differences of T and of
// V from there on.  So the barriers cut a mapping's simulation into
// independent segments: its makespan is the sum of its segments' makespans,
// each simulated on its own from time 0, and it is infeasible exactly when
// one of them is.  (The problem is §2.1's; serial workflows, fan-outs that
// join, and spines with fan-outs are cut this way, §4.1's diamonds among
// them.)  Segments of n_1, n_2, ... tools have 3^n_1 + 3^n_2 + ... mappings
// to simulate instead of 3^(n_1 + n_2 + ...).  An evaluation simulates them
// into tables and writes every whole mapping's makespan as a sum of entries;
// a branch and bound needs each segment's best only: the optimum is their sum,
// and its lowest index joins the segments' lowest.
#pragma once

#include <stdint.h>

#include "bf_lanetree.cuh"
#include "bf_plan.h"

namespace bfk {

constexpr uint32_t kSegMaxTools = 13;    // largest segment simulated whole (3^13 table entries, 6.4 MB)
constexpr uint32_t kSegMax = 32;         // segments of a scenario at most (one per tool)
// Table entry of an infeasible segment mapping, and the least sum that counts
// as infeasible: two of them add without a carry out of 32 bits.  Scenarios
// whose makespan bound reaches it keep the general kernels.
constexpr uint32_t kSegInfeasible = 0x7FFFFFFFu;

// The segments [start[j], start[j + 1]) of a scenario and what the kernels need
// to simulate them, passed by value with the launch.  A segment of two or more
// tools has a table in the handle's scratch, written anew by every call: the
// makespan of mapping m of segment j (its tools' digits, the first tool least
// significant) is entry off[j] + m.  Every entry is written once per call, and
// always with the same value, so calls of one handle whose GPU work overlaps
// do not disturb each other.  A one-tool segment's makespans are its tool's
// isolated times, alone[j].
struct SegPlan {
  uint32_t count;    // segments; 0: the scenario is not cut
  uint32_t tables;   // segments of two or more tools
  uint32_t entries;  // words of their tables
  uint32_t nmax;     // tools of the largest segment
  uint32_t budget;
  uint32_t start[kSegMax + 1];
  uint32_t size[kSegMax];  // 3^tools
  uint32_t off[kSegMax];
  uint32_t alone[kSegMax][3];
  // Tables: the segment, its lane-tree levels and its first block.
  uint32_t seg[kSegMax / 2], x[kSegMax / 2], y[kSegMax / 2], first_block[kSegMax / 2 + 1];
  // Tools, renumbered within each segment (a record's order), at its start.
  uint32_t pred[kSegMax], dur[3][kSegMax], vram[kSegMax], pv[kSegMax];
  uint32_t f[kSegMaxTools + 1];
  uint64_t frecip[kSegMaxTools + 1];
};

// What the evaluation's sums read: mappings [first, last] (canonical indices,
// n <= 20 tools), split at one barrier into low parts x in [0, A) -- the tools
// of segments [0, split) -- and rows h: index = x + A * h.
struct SegSums {
  uint32_t count, split, A;
  uint32_t first, last;
  uint32_t h_lo, h_hi;  // rows that hold an index of [first, last]
  uint32_t x_tiles, rows;  // tiled form: tiles of x, rows per block
  uint32_t size[kMaxTools], off[kMaxTools], alone[kMaxTools][3];
};

// The sums of the entries of segments [j0, j1) under the digits of each v[k]
// (segment j0 least significant), at most kSegInfeasible.  Entries are read
// through L2: the sum kernels may start before the tables are complete.
template <uint32_t K>
__device__ __forceinline__ void segment_sum(const SegSums& s, const uint32_t* table, uint32_t j0, uint32_t j1,
                                            uint32_t (&v)[K], uint32_t (&sum)[K]) {
#pragma unroll
  for (uint32_t k = 0; k < K; ++k) sum[k] = 0u;
  for (uint32_t j = j0; j < j1; ++j) {
    const uint32_t size = s.size[j];
#pragma unroll
    for (uint32_t k = 0; k < K; ++k) {
      const uint32_t q = v[k] / size, m = v[k] - q * size;
      const uint32_t t = size == 3u ? s.alone[j][m] : __ldcg(table + s.off[j] + m);
      sum[k] = sum[k] + t < kSegInfeasible ? sum[k] + t : kSegInfeasible;
      v[k] = q;
    }
  }
}

__device__ __forceinline__ uint32_t segment_sum(const SegSums& s, const uint32_t* table, uint32_t j0, uint32_t j1,
                                                uint32_t v) {
  uint32_t vs[1] = {v}, sum[1];
  segment_sum<1>(s, table, j0, j1, vs, sum);
  return sum[0];
}

namespace host {

// The scenario of tools [lo, hi) alone.
inline void segment_desc(const bf_scenario_desc* d, uint32_t lo, uint32_t hi, bf_scenario_desc* out) {
  std::memset(out, 0, sizeof *out);
  out->n = hi - lo;
  for (uint32_t j = 0; j < out->n; ++j) {
    out->pred_mask[j] = d->pred_mask[lo + j] >> lo;
    out->cpu_us[j] = d->cpu_us[lo + j];
    out->gpu_us[j] = d->gpu_us[lo + j];
    out->xfer_us[j] = d->xfer_us[lo + j];
    out->load_us[j] = d->load_us[lo + j];
    out->vram_mib[j] = d->vram_mib[lo + j];
  }
  out->vram_budget_mib = d->vram_budget_mib;
  std::memcpy(out->slowdown_q10, d->slowdown_q10, sizeof out->slowdown_q10);
}

// Blocks a table's roots are spread over at most: 5 on each of 152 SMs.
constexpr uint32_t kSegMaxBlocks = 760;

// The cut of a scenario (plan->count = 0 when it has no barrier, or a segment
// of more than kSegMaxTools tools, or makespans that may reach
// kSegInfeasible).  `bound` is the validator's makespan bound.
inline void segment_plan(const bf_scenario_desc* d, uint64_t bound, SegPlan* plan) {
  std::memset(plan, 0, sizeof *plan);
  const uint32_t n = d->n;
  if (bound >= kSegInfeasible) return;
  uint32_t anc[BF_MAX_TOOLS] = {};
  for (uint32_t v = 0; v < n; ++v) {
    anc[v] = d->pred_mask[v];
    for (uint32_t u = 0; u < v; ++u)
      if ((d->pred_mask[v] >> u) & 1u) anc[v] |= anc[u];
  }
  uint32_t count = 0;
  plan->start[0] = 0;
  for (uint32_t c = 1; c <= n; ++c) {
    const uint32_t below = c >= 32 ? ~0u : (1u << c) - 1u;
    bool barrier = true;
    for (uint32_t v = c; v < n; ++v) barrier = barrier && (anc[v] & below) == below;
    if (!barrier) continue;
    const uint32_t tools = c - plan->start[count];
    if (tools > kSegMaxTools) return;
    plan->nmax = tools > plan->nmax ? tools : plan->nmax;
    plan->size[count] = (uint32_t)pow3(tools);
    plan->start[++count] = c;
  }
  if (count < 2) return;
  plan->count = count;
  plan->budget = d->vram_budget_mib;
  for (uint32_t j = 0; j < count; ++j) {
    const uint32_t lo = plan->start[j], tools = plan->start[j + 1] - lo;
    bf_scenario_desc sd;
    segment_desc(d, lo, lo + tools, &sd);
    if (tools == 1u) {
      const bool fits = sd.vram_mib[0] <= sd.vram_budget_mib;
      plan->alone[j][0] = sd.cpu_us[0];
      plan->alone[j][1] = fits ? sd.gpu_us[0] + sd.xfer_us[0] : kSegInfeasible;
      plan->alone[j][2] = fits ? sd.load_us[0] + sd.gpu_us[0] + sd.xfer_us[0] : kSegInfeasible;
      continue;
    }
    // A root per lane as long as the GPU has lanes: the table launch is bound
    // by the latency of a lane's simulations, not by the issue rate.
    LaneTreeRecord r;
    const uint64_t most = (uint64_t)kSegMaxBlocks * 256u;
    lanetree_record(&sd, &r, plan->size[j] < most ? plan->size[j] : most);
    const uint32_t t = plan->tables++;
    const uint64_t want = (pow3(r.x) + 255u) / 256u;
    plan->seg[t] = j;
    plan->x[t] = r.x;
    plan->y[t] = r.y;
    plan->first_block[t + 1] = plan->first_block[t] + (uint32_t)(want < kSegMaxBlocks ? want : kSegMaxBlocks);
    plan->off[j] = plan->entries;
    plan->entries += plan->size[j];
    for (uint32_t v = 0; v < tools; ++v) {
      plan->pred[lo + v] = r.pred[v];
      for (uint32_t a = 0; a < 3; ++a) plan->dur[a][lo + v] = r.dur[a][v];
      plan->vram[lo + v] = r.vram[v];
      plan->pv[lo + v] = r.pv[v];
    }
    for (uint32_t k = 0; k <= tools; ++k) {
      plan->f[k] = r.f[k];
      plan->frecip[k] = r.frecip[k];
    }
  }
}

// Tiles of the sums: threads, and x values per thread.
constexpr uint32_t kSegThreads = 256, kSegPerThread = 8, kSegTile = kSegThreads * kSegPerThread;
constexpr uint32_t kSegMaxRows = 512;  // rows of a block (their sums are kept in shared memory)
constexpr uint32_t kSegDirect = 4;     // mappings per thread of the direct form

// Sums over mappings [first, first + count), count >= 1.  The split is the
// barrier nearest the middle, the later one of two: low parts wide enough to
// fill tiles, and as few sums of table entries as possible per block.  Below
// one tile of low parts the direct form runs (x_tiles = 0).
inline void segment_sums(const SegPlan& plan, uint64_t first, uint64_t count, SegSums* s) {
  std::memset(s, 0, sizeof *s);
  s->count = plan.count;
  const uint32_t n = plan.start[plan.count];
  uint32_t best = 0;
  for (uint32_t j = 1; j < plan.count; ++j) {
    const uint32_t c = plan.start[j], m = c < n - c ? c : n - c;
    if (m >= best) {
      best = m;
      s->split = j;
    }
  }
  s->A = (uint32_t)pow3(plan.start[s->split]);
  s->first = (uint32_t)first;
  s->last = (uint32_t)(first + count - 1);
  s->h_lo = s->first / s->A;
  s->h_hi = s->last / s->A;
  for (uint32_t j = 0; j < plan.count; ++j) {
    s->size[j] = plan.size[j];
    s->off[j] = plan.off[j];
    for (uint32_t a = 0; a < 3; ++a) s->alone[j][a] = plan.alone[j][a];
  }
  if (s->A >= kSegTile) {
    // About 8 blocks on each of 152 SMs; a warp takes a row at a time.
    s->x_tiles = (s->A + kSegTile - 1) / kSegTile;
    const uint32_t h = s->h_hi - s->h_lo + 1, chunks = (1216 + s->x_tiles - 1) / s->x_tiles;
    const uint32_t warps = kSegThreads / 32, rows = ((h + chunks - 1) / chunks + warps - 1) / warps * warps;
    s->rows = rows < kSegMaxRows ? rows : kSegMaxRows;
  }
}

}  // namespace host
}  // namespace bfk
