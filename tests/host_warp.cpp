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

#include "host_warp.h"

#include "../paper_2607_22242_gb300/csrc/bf_plan.h"

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
