"""Index-range searches on the lane tree (GPU): the range's ends inside every level, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2607_22242_gb300 import bf
from paper_2607_22242_gb300 import scenarios as S

THREADS = oracle.default_threads()


def _layered(n, seed, late_source):
    rng = np.random.default_rng(seed)
    base = S.random_small(rng, n, edge_p=0.0, tight=True, contention=True, max_time=9)
    pred = [0] * n
    for v in range(4, n):
        pred[v] = sum(1 << u for u in range((v // 4 - 1) * 4, v // 4 * 4) if rng.uniform() < 0.4) or 1 << (v - 4)
    if late_source:
        pred[n - 2] = 0  # the renumbered tools' indices are then not in the scenario's order
    return S.Scenario(**{**base.to_dict(), "pred_mask": pred})


@pytest.mark.gpu
@pytest.mark.parametrize("n", [10, 13, 17])
@pytest.mark.parametrize("late_source", [False, True])
def test_ranges_of_the_lane_tree(n, late_source):
    """The narrow form, at its smallest size too, and the wide one: whole spaces short of one mapping at either end,
    ranges cut at and beside the place values of single tools, and random ones of an eighth of the space or more."""
    scn = _layered(n, 31 + n, late_source)
    total = 3 ** n
    rng = np.random.default_rng(n)
    cuts = [3 ** (n - 1), 2 * 3 ** (n - 1), 3 ** (n - 1) + 3 ** (n - 2)]
    ranges = [(1, total - 1), (0, total - 1), (cuts[0], cuts[0]), (cuts[0] + 1, cuts[0]), (cuts[2] - 1, 3 ** (n - 1) + 2)]
    for _ in range(3):
        count = int(rng.integers(total // 8 + 1, total))
        ranges.append((int(rng.integers(0, total - count + 1)), count))
    with bf.create_scenario(scn) as h:
        for first, count in ranges if n < 17 else ranges[2:5]:
            want = oracle.search_range(scn, first, count, THREADS)
            for _ in range(2):  # the launch state resets itself
                r = bf.search_range(h, first, count)
                assert (r.index, r.makespan_us) == (want[0], want[1]), (first, count)
