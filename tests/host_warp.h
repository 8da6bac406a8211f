// One warp of a kernel on the CPU, for tests that run without a GPU: 32 lanes
// as coroutines that meet at the warp's collectives, and shared memory that
// promises no more than CUDA does -- a lane's stores are visible to the others
// only after a __syncwarp; votes, reductions and shuffles order no memory.
// Each lane works on a view of its own, and a __syncwarp copies every changed
// word to all views, so code that reads another lane's words without one reads
// stale words here every time.  Test infrastructure only.
#pragma once

#include <ucontext.h>

#include <cstdint>
#include <cstring>
#include <functional>
#include <vector>

struct HostDim {
  unsigned x;
};
static HostDim threadIdx{0}, blockDim{1};

namespace hostwarp {

constexpr unsigned kLanes = 32;
enum Op : int { kNone, kBallot, kShfl, kShflUp, kMax, kAdd, kSync };

struct Warp {
  ucontext_t scheduler, lane_ctx[kLanes];
  std::vector<char> stack[kLanes];
  Op op[kLanes];
  uint32_t value[kLanes], arg[kLanes], result[kLanes];
  bool done[kLanes];
  unsigned current = 0;
  std::function<void(unsigned)> body;
  std::vector<uint32_t> common;       // shared memory as of the last __syncwarp
  std::vector<uint32_t> view[kLanes]; // and as each lane sees it
  int error = 0;  // 1: lanes met at different collectives; 2: two lanes wrote one word between two __syncwarps
};
static Warp* g_warp = nullptr;

static void entry() {
  Warp& w = *g_warp;
  const unsigned lane = w.current;
  w.body(lane);
  w.done[lane] = true;
  swapcontext(&w.lane_ctx[lane], &w.scheduler);
}

static uint32_t meet(Op op, uint32_t value, uint32_t arg) {
  Warp& w = *g_warp;
  const unsigned lane = w.current;
  w.op[lane] = op;
  w.value[lane] = value;
  w.arg[lane] = arg;
  swapcontext(&w.lane_ctx[lane], &w.scheduler);
  return w.result[lane];
}

static void publish(Warp& w) {
  for (size_t i = 0; i < w.common.size(); ++i) {
    const uint32_t was = w.common[i];
    for (unsigned l = 0; l < kLanes; ++l) {
      if (w.view[l][i] == was) continue;
      if (w.common[i] != was && w.common[i] != w.view[l][i]) w.error = 2;
      w.common[i] = w.view[l][i];
    }
  }
  for (unsigned l = 0; l < kLanes; ++l) w.view[l] = w.common;
}

// Run body(lane) on the 32 lanes of one warp whose shared memory starts as
// `words`; 0, or Warp::error.
static int run(const std::vector<uint32_t>& words, std::function<void(unsigned)> body) {
  Warp w;
  g_warp = &w;
  w.body = body;
  w.common = words;
  for (unsigned l = 0; l < kLanes; ++l) {
    w.view[l] = words;
    w.stack[l].resize(1 << 18);
    w.done[l] = false;
    w.op[l] = kNone;
    getcontext(&w.lane_ctx[l]);
    w.lane_ctx[l].uc_stack.ss_sp = w.stack[l].data();
    w.lane_ctx[l].uc_stack.ss_size = w.stack[l].size();
    w.lane_ctx[l].uc_link = nullptr;
    makecontext(&w.lane_ctx[l], entry, 0);
  }
  for (;;) {
    unsigned left = 0;
    for (unsigned l = 0; l < kLanes; ++l) {
      if (w.done[l]) continue;
      w.op[l] = kNone;
      w.current = l;
      threadIdx.x = l;
      swapcontext(&w.scheduler, &w.lane_ctx[l]);
      left += w.done[l] ? 0u : 1u;
    }
    if (left == 0 || w.error) break;
    for (unsigned l = 0; l < kLanes; ++l)
      if (left != kLanes || w.op[l] != w.op[0]) w.error = 1;
    if (w.error) break;
    uint32_t ballot = 0, most = 0, sum = 0;
    for (unsigned l = 0; l < kLanes; ++l) {
      ballot |= w.value[l] ? 1u << l : 0u;
      most = w.value[l] > most ? w.value[l] : most;
      sum += w.value[l];
    }
    for (unsigned l = 0; l < kLanes; ++l) switch (w.op[l]) {
        case kBallot: w.result[l] = ballot; break;
        case kShfl: w.result[l] = w.value[w.arg[l] % kLanes]; break;
        case kShflUp: w.result[l] = w.value[l >= w.arg[l] ? l - w.arg[l] : l]; break;
        case kMax: w.result[l] = most; break;
        case kAdd: w.result[l] = sum; break;
        default: break;
      }
    if (w.op[0] == kSync) publish(w);
  }
  g_warp = nullptr;
  return w.error;
}

// This lane's view of the warp's shared memory.
static uint32_t* shared() { return g_warp->view[g_warp->current].data(); }

}  // namespace hostwarp

static inline uint32_t __ballot_sync(uint32_t, uint32_t p) { return hostwarp::meet(hostwarp::kBallot, p ? 1u : 0u, 0u); }
static inline uint32_t __shfl_sync(uint32_t, uint32_t v, uint32_t from) { return hostwarp::meet(hostwarp::kShfl, v, from); }
static inline uint32_t __shfl_up_sync(uint32_t, uint32_t v, uint32_t o) { return hostwarp::meet(hostwarp::kShflUp, v, o); }
static inline uint32_t __reduce_max_sync(uint32_t, uint32_t v) { return hostwarp::meet(hostwarp::kMax, v, 0u); }
static inline uint32_t __reduce_add_sync(uint32_t, uint32_t v) { return hostwarp::meet(hostwarp::kAdd, v, 0u); }
static inline void __syncwarp() { hostwarp::meet(hostwarp::kSync, 0u, 0u); }
