"""The tree search's chains of levels and its leaf modes (GPU): every optimum is the oracle's, ties included, whatever
bound the search starts from."""
import numpy as np
import pytest

import oracle
from paper_2607_22242_gb300 import bf
from paper_2607_22242_gb300 import scenarios as S

THREADS = oracle.default_threads()


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 5, 6, 9, 10, 13, 14])
def test_optima_from_any_bound(n):
    """No level above the leaves (5 tools and fewer), one start level only (1 to 243 leaf nodes, cut into parts of 2
    combinations and more), start and expansions, and dives (14 tools): hints at the optimum (the tightest bound that
    keeps it), at another mapping and none; small times, so that ties are frequent, tight budgets, late sources, a last
    tool that waits for all others."""
    rng = np.random.default_rng(n)
    for t in range(8 if n < 13 else 4 if n < 14 else 2):
        base = S.random_small(rng, n, edge_p=float(rng.choice([0.1, 0.4])), tight=bool(t % 3), contention=bool(t % 4),
                              max_time=int(rng.choice([3, 9, 60])))
        pred = list(base.pred_mask)
        if t % 3 == 0 and n > 3:
            pred[n - 2] = 0
        if t % 4 == 1 and n > 2:
            pred[n - 1] = (1 << (n - 1)) - 1
        scn = S.Scenario(**{**base.to_dict(), "pred_mask": pred})
        full, binary = oracle.search(scn, THREADS), oracle.search_binary(scn, THREADS)
        with bf.create_scenario(scn) as h:
            for space, want in ((bf.SPACE_FULL, full), (bf.SPACE_BINARY, binary)):
                for hint in (None, want[0], int(rng.integers(0, 3 ** n))):
                    r, stats = bf.search_tree(h, space, True, hint)
                    assert (r.index, r.makespan_us) == want, (t, space, hint)
                    assert stats["leaves"] <= space ** n * 3  # at most every mapping in each dive and the search
                r, _ = bf.search_tree(h, space, False)
                assert (r.index, r.makespan_us) == want, (t, space)
