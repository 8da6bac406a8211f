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
