"""Device code whose lanes read each other's shared memory, on a CPU warp without memory ordering between
__syncwarps (tests/host_warp.h), against the oracle (no GPU)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_2607_22242_gb300 import bf
from paper_2607_22242_gb300 import scenarios as S

HERE = os.path.dirname(os.path.abspath(__file__))
THREADS = oracle.default_threads()


@pytest.fixture(scope="module")
def warp(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("warp") / "host_warp.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-Wno-unknown-pragmas", "-I",
                    os.path.join(HERE, "..", "include"), "-o", out, os.path.join(HERE, "host_warp.cpp")], check=True)
    lib = ctypes.CDLL(out)
    lib.host_lanetree_warp.argtypes = [ctypes.POINTER(bf.Desc), ctypes.c_uint32, ctypes.c_uint32, ctypes.c_int,
                                       ctypes.c_void_p, ctypes.c_void_p]
    lib.host_lanetree_warp.restype = ctypes.c_int
    lib.host_leaf_warps.argtypes = [ctypes.POINTER(bf.Desc), ctypes.c_uint32, ctypes.c_int, ctypes.c_uint32,
                                    ctypes.c_uint32, ctypes.c_void_p, ctypes.c_void_p]
    lib.host_leaf_warps.restype = ctypes.c_int
    return lib


@pytest.mark.parametrize("n,x,y", [(5, 1, 3), (7, 1, 4), (7, 2, 4), (8, 3, 7), (8, 4, 8)])
@pytest.mark.parametrize("wide", [False, True])
def test_lanes_take_over_combinations(warp, n, x, y, wide):
    """Fewer roots than lanes, and a few more (three levels and two): every feasible mapping reported once with the
    oracle's makespan, most of them by lanes that took over another's combinations."""
    rng = np.random.default_rng(n * 100 + x * 10 + y)
    shared = np.zeros(1, np.uint32)
    taken = 0
    for t in range(4):
        scn = S.random_small(rng, n, edge_p=float(rng.choice([0.1, 0.4])), tight=bool(t % 2), contention=True,
                             max_time=int(rng.choice([5, 40])))
        got = np.zeros(3 ** n, np.uint32)
        assert warp.host_lanetree_warp(ctypes.byref(bf.to_desc(scn)), x, y, int(wide), got.ctypes.data,
                                       shared.ctypes.data) == 0
        want, _ = oracle.eval_range(scn, 0, 3 ** n, THREADS)
        bad = np.flatnonzero(got.astype(np.uint64) != want)
        assert bad.size == 0, (t, bad.size, int(bad[0]))
        taken += int(shared[0])
    assert taken > 0


def _leaves(warp, scn, space, start, bounds, prune=True):
    """((index, makespan), mappings simulated, nodes of the first tasks, leaf nodes) of the leaf tasks."""
    out, b = np.zeros(5, np.uint64), np.array(bounds, np.uint32)
    assert warp.host_leaf_warps(ctypes.byref(bf.to_desc(scn)), space, int(prune), start, b.size, b.ctypes.data,
                                out.ctypes.data) == 0
    ms, idx = int(out[0]), int(out[1])
    return (idx, ms) if ms != 2 ** 64 - 1 else (-1, 0xFFFFFFFF), int(out[2]), int(out[3]), int(out[4])


@pytest.mark.parametrize("n", [6, 8, 10])
@pytest.mark.parametrize("parts", [1, 3, 16])
def test_leaf_tasks_share_nodes(warp, n, parts):
    """Leaf groups from no bound (every lane on its own node), from just above the optimum and at it (few
    combinations, dealt over the lanes, which read one another's states), and unpruned: the oracle's optimum."""
    rng = np.random.default_rng(n)
    for t in range(3):
        scn = S.random_small(rng, n, edge_p=0.3, tight=bool(t % 2), contention=True, max_time=(9, 60, 500)[t])
        for space, want in ((3, oracle.search(scn, THREADS)), (2, oracle.search_binary(scn, THREADS))):
            for start in (0xFFFFFFFF, want[1] + want[1] // 10, want[1]):
                got = _leaves(warp, scn, space, start, [start] * parts)
                assert got[0] == want, (t, space, start, got, want)
            if n <= 8:
                assert _leaves(warp, scn, space, 0xFFFFFFFF, [0xFFFFFFFF] * parts, prune=False)[0] == want


def _layered(n, seed):
    """A layered DAG (layers of 4, edge probability 0.4) with the standard profile recipe, 24 GiB."""
    rng = np.random.default_rng(seed)
    c, g, x, m = S._ordinary(np.random.default_rng([seed, n]), n, 2048, 16384)
    pred = S._layered_edges(rng, [4] * (n // 4) + ([n % 4] if n % 4 else []), 0.4)
    return S.Scenario(n, pred, c, g, x, [S._load_from_vram(v) for v in m], m, 24576, S.slowdown_linear(kmax=n))


@pytest.mark.parametrize("n,seed,parts", [(11, 0, 5), (11, 0, 16), (12, 1, 2), (12, 1, 5), (12, 1, 16), (13, 3, 2)])
def test_leaf_tasks_while_the_bound_improves(warp, n, seed, parts):
    """The best makespan improves between the tasks of a node group, at every place among them (from 5 % above the
    optimum to the optimum): the optimum is found all the same, and the tasks simulate as many combinations in all as
    without the improvement -- the parts stay those of one list."""
    scn = _layered(n, seed)
    opt = oracle.search(scn, THREADS)
    loose = opt[1] + opt[1] // 20
    want = _leaves(warp, scn, 3, loose, [loose] * parts)
    assert want[0] == opt
    for k in range(parts + 1):
        got = _leaves(warp, scn, 3, loose, [loose] * k + [opt[1]] * (parts - k))
        assert got[0] == opt, k
        assert got[1:] == want[1:], k
