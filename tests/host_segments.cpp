// Host build of the cut at barriers (bf_segments.cuh) for tests that run
// without a GPU: the segments' tables are simulated with the lane tree's code
// and every mapping's makespan is the sum the evaluation kernels form.  Test
// infrastructure only; the library never runs this.
#include <algorithm>
#include <cstdint>
#include <cstring>
#include <vector>

#define __device__
#define __host__
#define __forceinline__ inline
using std::min;
static inline int __popc(unsigned x) { return __builtin_popcount(x); }
static inline int __ffs(unsigned x) { return __builtin_ffs((int)x); }
static inline uint32_t __ldcg(const uint32_t* p) { return *p; }
struct HostDim {
  unsigned x;
};
static HostDim threadIdx{0}, blockDim{1};

#include "../paper_2607_22242_gb300/csrc/bf_segments.cuh"

using namespace bfk;

namespace {
struct Store {
  uint32_t* table;
  uint64_t* writes;
  void operator()(uint32_t idx, uint32_t ms) { table[idx] = ms; ++*writes; }
  void dead(uint32_t idx) { table[idx] = kSegInfeasible; ++*writes; }
};
}  // namespace

// The plan's segments (start[0 .. count]); 0 when the scenario is not cut.
// `bound` is the makespan bound the plan is given.  With out[], every mapping
// of [first, first + count): its makespan, 0xFFFFFFFF if infeasible.
extern "C" uint32_t host_segments(const bf_scenario_desc* d, uint64_t bound, uint64_t first, uint64_t count,
                                  uint32_t* out, uint32_t* start) {
  static SegPlan plan;
  host::segment_plan(d, bound, &plan);
  for (uint32_t j = 0; j <= plan.count; ++j) start[j] = plan.start[j];
  if (plan.count == 0u || !out) return plan.count;
  std::vector<uint32_t> table(plan.entries + 1u, 0xDEADBEEFu);
  threadIdx.x = 0;
  blockDim.x = 1;
  for (uint32_t t = 0; t < plan.tables; ++t) {
    const uint32_t seg = plan.seg[t], lo = plan.start[seg], n = plan.start[seg + 1] - lo;
    std::vector<LtSharedT<3>> shared(1);
    LtSharedT<3>& S = shared[0];
    std::memset(&S.rec, 0, sizeof S.rec);
    S.rec.n = n;
    S.rec.budget = plan.budget;
    S.rec.all_mask = (1u << n) - 1u;
    S.rec.x = plan.x[t];
    S.rec.y = plan.y[t];
    for (uint32_t v = 0; v < n; ++v) {
      S.rec.pred[v] = plan.pred[lo + v];
      for (uint32_t a = 0; a < 3; ++a) S.rec.dur[a][v] = plan.dur[a][lo + v];
      S.rec.vram[v] = plan.vram[lo + v];
      S.rec.pv[v] = plan.pv[lo + v];
      S.rec.big_mask |= plan.vram[lo + v] > plan.budget ? 1u << v : 0u;
    }
    for (uint32_t k = 0; k <= n; ++k) {
      S.rec.f[k] = plan.f[k];
      S.rec.frecip[k] = plan.frecip[k];
    }
    lt_fill_tables(S);
    std::vector<uint32_t> rows(lt_rows<false>(n), 0xA5A5A5A5u);
    uint64_t writes = 0;
    Store sink{table.data() + plan.off[seg], &writes};
    uint32_t next = 0, roots = (uint32_t)host::pow3(S.rec.x);
    lt_lane<3, false, true>(S, rows.data(), 1u, [&]() { return next < roots ? next++ : 0xFFFFFFFFu; }, sink);
    if (writes != plan.size[seg]) return 0xFFFFFFFFu;  // every entry is written once
  }
  SegSums sums;
  host::segment_sums(plan, first, count, &sums);
  for (uint64_t i = 0; i < count; ++i) {
    const uint32_t idx = (uint32_t)(first + i), h = idx / sums.A;
    if (h < sums.h_lo || h > sums.h_hi) return 0xFFFFFFFEu;
    const uint32_t sum = segment_sum(sums, table.data(), 0u, sums.split, idx - h * sums.A) +
                         segment_sum(sums, table.data(), sums.split, sums.count, h);
    out[i] = sum < kSegInfeasible ? sum : 0xFFFFFFFFu;
  }
  return plan.count;
}
