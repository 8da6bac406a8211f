"""Scenarios cut by barriers: the cut and its sums on the host, the evaluation and optimum kernels on the GPU, all
against the oracle (whole microseconds: nothing may differ)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
from oracle import segments
from paper_2607_22242_gb300 import bf
from paper_2607_22242_gb300 import scenarios as S

HERE = os.path.dirname(os.path.abspath(__file__))
THREADS = oracle.default_threads()


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("segments") / "host_segments.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(HERE, "..", "include"), "-o",
                    out, os.path.join(HERE, "host_segments.cpp")], check=True)
    lib = ctypes.CDLL(out)
    lib.host_segments.argtypes = [ctypes.POINTER(bf.Desc), ctypes.c_uint64, ctypes.c_uint64, ctypes.c_uint64,
                                  ctypes.c_void_p, ctypes.c_void_p]
    lib.host_segments.restype = ctypes.c_uint32

    def run(scn, first=0, count=0, bound=1 << 30):
        start = np.zeros(33, np.uint32)
        ms = np.zeros(count, np.uint32)
        n = lib.host_segments(ctypes.byref(bf.to_desc(scn)), bound, first, count,
                              ms.ctypes.data if count else None, start.ctypes.data)
        return start[:n + 1].tolist() if n < 64 else n, ms.astype(np.uint64)
    return run


def _barriers(scn):
    """Every c such that all tools >= c have all tools < c among their ancestors, from the definition."""
    anc = []
    for v in range(scn.n):
        a = scn.pred_mask[v]
        for u in range(v):
            if a >> u & 1:
                a |= anc[u]
        anc.append(a)
    return [c for c in range(1, scn.n) if all(anc[v] & ((1 << c) - 1) == (1 << c) - 1 for v in range(c, scn.n))]


@pytest.mark.parametrize("n,seg_max", [(2, 1), (3, 2), (6, 1), (7, 5), (9, 4), (11, 9)])
@pytest.mark.parametrize("tight", [False, True])
def test_sums_equal_simulations(host, n, seg_max, tight):
    """Random segmented DAGs: the cut is at every barrier and every mapping of the space and of ragged ranges is the
    oracle's."""
    rng = np.random.default_rng(n * 10 + seg_max)
    for _ in range(6):
        scn = S.random_segmented(rng, n, seg_max=seg_max, tight=tight)
        cuts = _barriers(scn)
        total = 3 ** n
        first = int(rng.integers(0, total))
        for f, c in ((0, total), (first, int(rng.integers(1, total - first + 1)))):
            start, ms = host(scn, f, c)
            if not cuts:
                assert start == [0]
                continue
            assert start == [0] + cuts + [n]
            want, _ = oracle.eval_range(scn, f, c, THREADS)
            assert np.array_equal(ms, want)


def test_scenarios_that_are_not_cut(host):
    """No barrier, a segment of more than 13 tools, or a makespan bound the tables' 31 bits cannot hold."""
    fan = lambda n: S.Scenario(n, [0] + [1] * (n - 2) + [(1 << (n - 1)) - 2], [9] * n, [5] * n, [0] * n, [1] * n,
                               [1] * n, 99, S.slowdown_linear(kmax=32))
    assert host(fan(15))[0] == [0, 1, 14, 15]
    assert host(fan(16))[0] == [0]
    assert host(fan(15), bound=0x7FFFFFFF)[0] == [0]
    assert host(S.layered24())[0] == [0]
    assert host(S.config3())[0] == [0, 1, 2, 9, 10, 11, 18, 19]


def _segmented(n, seg_max, seed, tight=True):
    rng = np.random.default_rng(seed)
    while True:
        scn = S.random_segmented(rng, n, seg_max=seg_max, tight=tight)
        if len(_barriers(scn)) >= 1:
            return scn


@pytest.mark.gpu
@pytest.mark.parametrize("n,seg_max,phase", [
    (4, 1, (0, 0)),    # no tables: one-tool segments only, one block
    (11, 1, (0, 0)),   # direct sums over several blocks
    (14, 1, (0, 0)),   # tiles: 3^7 low parts, just over one tile of 2,048
    (13, 7, (1, 1)),   # output arrays off the vectors' alignment by the same phase
    (13, 7, (2, 3)),   # and by different ones: mapping by mapping
    (14, 8, (3, 3)),
])
def test_evaluation_by_sums(n, seg_max, phase):
    """Whole spaces and ranges cut inside rows, tiles and vectors, into arrays at several alignments, with nothing
    written outside them."""
    import torch
    scn = _segmented(n, seg_max, seed=n * seg_max)
    total = 3 ** n
    want, feas = oracle.eval_range(scn, 0, total, THREADS)
    rng = np.random.default_rng(7)
    ranges = [(0, total), (1, total - 1), (0, total - 1)]
    ranges += [(int(f), int(rng.integers(min(total - f, 1 << 17), total - f + 1))) for f in rng.integers(0, total // 2, 4)]
    with bf.create_scenario(scn) as h:
        for first, count in ranges:
            ms = torch.full((count + 8,), 77, dtype=torch.int32, device="cuda")
            fe = torch.full((count + 8,), 9, dtype=torch.uint8, device="cuda")
            a, b = phase
            bf.eval_mappings(h, first, count, ms[a:a + count], fe[b:b + count])
            m, f = ms.cpu().numpy(), fe.cpu().numpy()
            assert np.array_equal(m[a:a + count].view(np.uint32), want[first:first + count].astype(np.uint32)), (first, count)
            assert np.array_equal(f[b:b + count], feas[first:first + count]), (first, count)
            assert (m[:a] == 77).all() and (m[a + count:] == 77).all() and (f[:b] == 9).all() and (f[b + count:] == 9).all()


@pytest.mark.gpu
def test_evaluations_of_one_handle_overlap():
    """Evaluations of one handle on two streams at once share its tables: both are right."""
    import torch
    scn = S.config3()
    first, count = 400_000_001, 1 << 22
    with bf.create_scenario(scn) as h:
        streams = [torch.cuda.Stream() for _ in range(2)]
        outs = []
        for k in range(8):
            outs.append(bf.eval_mappings(h, first, count, stream=streams[k % 2]))
        torch.cuda.synchronize()
        want, _ = oracle.eval_range(scn, first, 4096, THREADS)
        for ms, _ in outs:
            assert torch.equal(ms, outs[0][0])
            assert np.array_equal(ms[:4096].cpu().numpy().view(np.uint32), want.astype(np.uint32))


@pytest.mark.gpu
def test_captured_evaluation_outlives_its_handle():
    """An evaluation captured into a graph with a temporary handle runs after the handle is gone."""
    import torch
    scn = S.config1()
    total = 3 ** scn.n
    ms = torch.zeros(total, dtype=torch.int32, device="cuda")
    fe = torch.zeros(total, dtype=torch.uint8, device="cuda")
    bf.eval_mappings(scn, 0, total, ms, fe)  # loads the kernels
    want, flags = ms.clone(), fe.clone()
    h = bf.create_scenario(scn)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        bf.eval_mappings(h, 0, total, ms, fe)
    h.close()
    ms.zero_()
    fe.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(ms, want) and torch.equal(fe, flags)


@pytest.mark.gpu
def test_first_evaluation_beside_a_capture():
    """A handle's first evaluation (which allocates its tables) on one stream while another stream is being captured:
    the capture goes on, and both give the right values."""
    import torch
    scn = S.config3()
    first, count = 400_000_001, 1 << 18
    x = torch.zeros(4, device="cuda")
    want = bf.eval_mappings(scn, first, count)  # loads the kernels
    ms = torch.zeros(count, dtype=torch.int32, device="cuda")
    fe = torch.zeros(count, dtype=torch.uint8, device="cuda")
    other = torch.cuda.Stream()
    torch.cuda.synchronize()
    with bf.create_scenario(scn) as h:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            x.add_(1)
            bf.eval_mappings(h, first, count, ms, fe, stream=other)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(ms, want[0]) and torch.equal(fe, want[1]) and (x == 1).all()


@pytest.mark.gpu
@pytest.mark.parametrize("n,seg_max", [(2, 1), (9, 9), (20, 1), (32, 1), (32, 8), (27, 13)])
def test_optimum_by_segments(n, seg_max):
    """Branch and bound over both spaces of scenarios cut by barriers, twice on one handle (the launch state resets
    itself), against the oracle's segment rule."""
    scn = _segmented(n, seg_max, seed=n + seg_max)
    with bf.create_scenario(scn) as h:
        for space, binary in ((bf.SPACE_FULL, False), (bf.SPACE_BINARY, True)):
            want = segments.search(scn, binary=binary, threads=THREADS)
            for _ in range(2):
                r, stats = bf.search_tree(h, space)
                assert (r.index, r.makespan_us, r.feasible) == (want[0], want[1], True)
                assert stats["leaves"] <= space ** n
            if n <= 20 and not binary:
                r = bf.search_pruned(h)
                assert (r.index, r.makespan_us) == want
