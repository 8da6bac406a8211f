"""The lane tree's closed-form endings and the virtual-clock advance, at the values where they can go wrong (no GPU).

The kernels' code (bf_lanetree.cuh, bf_sim.cuh) is built for the host; whole results come from the oracle."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2607_22242_gb300 import scenarios as S
from test_host_enumeration import HERE, _same_lanetree, host  # noqa: F401  (host is a fixture)

ADVANCE = r"""
#include <cstdint>
#define __device__
#define __host__
#define __forceinline__ inline
#include <algorithm>
using std::min;
static inline int __popc(unsigned x) { return __builtin_popcount(x); }
static inline int __ffs(unsigned x) { return __builtin_ffs((int)x); }
struct HostDim { unsigned x; };
static HostDim threadIdx{0}, blockDim{1};
#include "../paper_2607_22242_gb300/csrc/bf_sim.cuh"
// The number of (dt, f) with f in [lo, hi) whose advance differs from the exact floor(dt 2^20 / f); only quotients
// of 32 bits are used (the advance is below a running tool's remaining work).
extern "C" uint64_t wrong(uint32_t lo, uint32_t hi, const uint32_t* dts, uint32_t n) {
  uint64_t bad = 0;
  for (uint32_t f = lo; f < hi; ++f)
    for (uint32_t j = 0; j < n; ++j)
      for (int64_t off = -2; off <= 2; ++off) {
        // dt itself, and the dt around each multiple of f (where the quotient steps)
        const uint64_t around = ((uint64_t)dts[j] * f >> 20) + (uint64_t)off;
        for (uint64_t dt : {(uint64_t)dts[j], around}) {
          if (dt > 0xFFFFFFFFull) continue;
          const uint64_t want = (dt << 20) / f;
          if (want > 0xFFFFFFFFull) continue;
          bad += bfk::cpu_advance((uint32_t)dt, f, (1ull << 52) / f) != (uint32_t)want;
        }
      }
  return bad;
}
"""


@pytest.mark.parametrize("lo,hi", [(1024, 1030), (1024, 65537)])
def test_cpu_advance_is_the_exact_floor(tmp_path, lo, hi):
    """Every slowdown in [lo, hi), with dt at the ends of its range, at powers of two and at random."""
    out = str(tmp_path / "advance.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", HERE, "-x", "c++", "-", "-o", out],
                   input=ADVANCE.replace('"../', '"%s/../' % HERE).encode(), check=True)
    lib = ctypes.CDLL(out)
    lib.wrong.restype = ctypes.c_uint64
    rng = np.random.default_rng(1)
    count = 4000 if hi - lo < 10 else 24
    dts = np.concatenate([[0, 1, 2, 1023, 1024, 2 ** 22 - 1, 2 ** 28, 2 ** 32 - 1],
                          2 ** rng.integers(0, 32, 8), rng.integers(0, 2 ** 32, count)]).astype(np.uint32)
    assert lib.wrong(lo, hi, dts.ctypes.data_as(ctypes.c_void_p), dts.size) == 0


def _scenario(n, pred, budget, vram, rng, steep):
    draw = lambda lo, hi: [int(v) for v in rng.integers(lo, hi, n)]
    slow = [0, 1024] + [1024 + k * (37 if steep else 0) * 13 for k in range(1, 20)]
    return S.Scenario(n, pred, draw(1, 60), draw(1, 30), draw(0, 5), draw(0, 20), vram, budget, slow)


@pytest.mark.parametrize("n", [1, 2, 5, 9])
@pytest.mark.parametrize("ending", ["drain", "blocked", "oversized", "joined"])
@pytest.mark.parametrize("wide", [False, True])
def test_endings_in_closed_form(host, n, ending, wide):  # noqa: F811
    """Every mapping of scenarios whose simulations end with one GPU tool: a queue draining beside CPU tools, a head
    blocked by the last running gpu_now tool, a waiting tool larger than the budget, and a last tool that waits for
    all others (nothing is settled before it starts)."""
    rng = np.random.default_rng(len(ending) * 100 + n)
    for steep in (False, True):
        vram = [int(v) for v in rng.integers(1, 6, n)]
        pred = [0] * n
        if ending == "joined" and n > 1:
            pred[-1] = (1 << (n - 1)) - 1
        budget = {"drain": 6 * n, "blocked": max(vram), "oversized": 4, "joined": 9}[ending]
        _same_lanetree(host, _scenario(n, pred, budget, vram, rng, steep), 3, 3 ** max(0, n - 6) if wide else 0, wide=wide)
