"""Handles made and destroyed one after the other, and by several threads at once, share pooled scratch (GPU); the
pool's own rules without one."""
import ctypes
import os
import subprocess
import threading

import pytest

import oracle
from paper_2607_22242_gb300 import bf
from paper_2607_22242_gb300 import scenarios as S


@pytest.mark.gpu
@pytest.mark.parametrize("threads,rounds", [(1, 40), (6, 25)])
def test_handles_in_turn(threads, rounds):
    """More handles than the pool keeps, of every kind of search, each result the oracle's: no launch state or record
    of an earlier handle is left in the scratch of a later one."""
    import numpy as np
    import torch
    rng = np.random.default_rng(threads)
    scns = [S.random_small(rng, int(n), edge_p=0.3) for n in rng.integers(2, 11, 12)]
    scns += [S.random_segmented(rng, 9), S.config0()]
    want = [oracle.search(s) for s in scns]
    errors = []

    def work(t):
        try:
            stream = torch.cuda.Stream()
            held = []
            for k in range(rounds):
                j = (k * 5 + t) % len(scns)
                h = bf.create_scenario(scns[j])
                held.append(h)
                for r in (bf.search_best(h, stream), bf.search_pruned(h, None, stream),
                          bf.search_tree(h, bf.SPACE_FULL, True, None, stream)[0]):
                    if (r.index, r.makespan_us) != want[j]:
                        errors.append((t, k, j, r))
                if len(held) > 4:
                    held.pop(0).close()
            for h in held:
                h.close()
        except Exception as e:  # noqa: BLE001
            errors.append((t, e))
    ts = [threading.Thread(target=work, args=(t,)) for t in range(threads)]
    for t in ts:
        t.start()
    for t in ts:
        t.join(timeout=120)
    assert not any(t.is_alive() for t in ts) and errors == []


@pytest.mark.gpu
def test_a_handle_closed_after_a_timeout_keeps_its_scratch_to_itself():
    """A one-off search whose wait runs out closes its handle with the kernel still running: the next handles get
    other scratch, and their results are right."""
    import torch
    scn, small = S.config3(), S.config0()
    bf.set_wait_timeout_ms(1)
    try:
        with pytest.raises(bf.BfError) as ei:
            bf.search_best(scn)
        assert ei.value.code == bf.BF_ETIMEOUT
        bf.set_wait_timeout_ms(600000)
        for _ in range(3):
            r = bf.search_best(small)
            assert (r.index, r.makespan_us) == oracle.search(small)
    finally:
        bf.set_wait_timeout_ms(600000)
        torch.cuda.synchronize()


HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def pool(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("pool") / "host_pool.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-o", out, os.path.join(HERE, "host_pool.cpp")],
                   check=True)
    return ctypes.CDLL(out)


@pytest.mark.parametrize("calls,may", [(b"", 1), (b"be", 1), (b"bebe", 1), (b"b", 0),
                                       (b"bbe", 0),      # a good call after one that stopped waiting
                                       (b"bebbebe", 0)])
def test_scratch_of_an_unfinished_call_is_never_kept(pool, calls, may):
    assert pool.host_may_keep(calls) == may


def test_pairs_stay_in_the_context_they_were_made_in(pool):
    """A pair is handed out only where it was made, also when its handle is destroyed under another context (after a
    device reset, say): such a pair is not kept at all, nor one whose context could not be told."""
    pool.host_keep.argtypes = [ctypes.c_void_p, ctypes.c_uint64, ctypes.c_uint64]
    pool.host_take.argtypes, pool.host_take.restype = [ctypes.c_uint64], ctypes.c_void_p
    assert pool.host_keep(16, 1, 1) == 1
    assert pool.host_keep(32, 1, 2) == 0
    assert pool.host_keep(48, 0, 2) == 0 and pool.host_keep(48, 0, 0) == 0
    assert pool.host_take(2) is None and pool.host_take(0) is None
    assert pool.host_take(1) == 16 and pool.host_take(1) is None
    kept = [pool.host_keep(16 * k, 3, 3) for k in range(1, 40)]
    assert sum(kept) == 16  # bounded


@pytest.mark.gpu
def test_a_good_call_after_a_timeout_does_not_release_the_scratch():
    """A search whose wait ran out, then a good call on another stream beside it: closing the handle waits for the
    search instead of handing its scratch on, and the next handles' results are right."""
    import torch
    scn, small = S.config3(), S.config0()
    slow, fast = torch.cuda.Stream(), torch.cuda.Stream(priority=-1)
    beside = 0
    try:
        for _ in range(5):
            h = bf.create_scenario(scn)
            bf.set_wait_timeout_ms(1)
            with pytest.raises(bf.BfError) as ei:
                bf.search_best(h, slow)
            assert ei.value.code == bf.BF_ETIMEOUT
            bf.set_wait_timeout_ms(600000)
            bf.whatif(h, 0, stream=fast)
            beside += not slow.query()  # the search was still running when the good call ended
            h.close()
            assert slow.query()
            r = bf.search_best(small)
            assert (r.index, r.makespan_us) == oracle.search(small)
    finally:
        bf.set_wait_timeout_ms(600000)
        torch.cuda.synchronize()
    assert beside > 0
