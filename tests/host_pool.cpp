// Host build of the scratch pool and of a handle's record of calls
// (bf_scratch_pool.h), driven from tests that run without a GPU.  Test
// infrastructure only.
#include "../paper_2607_22242_gb300/csrc/bf_scratch_pool.h"

using namespace bfcapi;

// Calls of one handle, in turn: 'b' puts work out, 'e' sees the end of the
// last such work.  1 when the handle's scratch may be kept for others.
extern "C" int host_may_keep(const char* calls) {
  OpenCalls c{};
  for (; *calls; ++calls) {
    if (*calls == 'b') c.begin();
    else c.end();
  }
  return c.none_open() ? 1 : 0;
}

static unsigned long long g_context;  // 0: none is current
static ScratchPool<int>& pool() {
  static ScratchPool<int> p([](unsigned long long* id) {
    *id = g_context;
    return g_context != 0;
  });
  return p;
}

// Give the pool a pair named `name` that was made in context `made_in` while
// `current` is; 1 when it was kept.
extern "C" int host_keep(int* name, unsigned long long made_in, unsigned long long current) {
  g_context = current;
  return pool().keep({name, name}, made_in) ? 1 : 0;
}

// The pair handed out while `current` is the context, or null.
extern "C" int* host_take(unsigned long long current) {
  g_context = current;
  ScratchPool<int>::Pair p;
  return pool().take(&p) ? p.d : nullptr;
}
