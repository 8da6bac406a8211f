"""Lanes that take over part of another lane's level-1 combinations (GPU): searches whose blocks hand out few roots, so
that most of the work is shared, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2607_22242_gb300 import bf
from paper_2607_22242_gb300 import scenarios as S

THREADS = oracle.default_threads()


def _uneven(rng, n):
    """A few early tools decide how much there is to simulate: half of their mappings run out of memory at once."""
    base = S.random_small(rng, n, edge_p=0.25, tight=True, contention=True, max_time=20)
    vram = list(base.vram_mib)
    vram[:3] = [base.vram_budget_mib] * 3
    return S.Scenario(**{**base.to_dict(), "vram_mib": vram})


@pytest.mark.gpu
@pytest.mark.parametrize("n", [7, 9, 10, 12, 13, 16, 17])
@pytest.mark.parametrize("count", [1, 5])
def test_batches_with_few_roots(n, count):
    """One and a few scenarios of each table form: the least roots per block, three levels and two."""
    rng = np.random.default_rng(n * 7 + count)
    scns = [_uneven(rng, n) for _ in range(count if n < 16 else 1)]
    idx, ms = oracle.search_batch(scns, THREADS) if n < 16 else ([], [])
    for _ in range(2):
        got = [(r.index, r.makespan_us) for r in bf.search_batch(scns)]
        if n < 16:
            assert got == list(zip(idx.tolist(), ms.tolist()))
        else:  # the same optimum from branch and bound
            assert got == [(r.index, r.makespan_us) for r in (bf.search_tree(s)[0] for s in scns)]


@pytest.mark.gpu
@pytest.mark.parametrize("n", [10, 12, 14])
def test_whole_space_searches_with_uneven_roots(n):
    rng = np.random.default_rng(n)
    for _ in range(3):
        scn = _uneven(rng, n)
        with bf.create_scenario(scn) as h:
            for _ in range(2):
                r = bf.search_best(h)
                assert (r.index, r.makespan_us) == oracle.search(scn, THREADS)
