"""Lists of mappings at the edges of the list kernel's forms (GPU), against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2607_22242_gb300 import bf
from paper_2607_22242_gb300 import scenarios as S


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 4, 12, 13, 16, 17, 20, 21, 25, 32])
@pytest.mark.parametrize("count", [1, 33, 5000])
def test_lists(n, count):
    """The largest and smallest scenario of each form, without edges: all n tools can wait in the queue at once (its
    second word holds the 13th, its third the 25th).  One mapping, a ragged warp, several blocks; indices at both ends
    of the space and beside it."""
    import torch
    rng = np.random.default_rng(n)
    scn = S.random_small(rng, n, edge_p=0.0, tight=n % 2 == 0, contention=True, max_time=30)
    total = 3 ** n
    idx = rng.integers(0, total, count, dtype=np.int64)
    edges = [total - 1, 0, 3 ** (n - 1), total, 2 ** 62, -1][:count]
    idx[:len(edges)] = edges
    ms, fe = bf.eval_indices(scn, torch.from_numpy(idx).cuda())
    ms, fe = ms.cpu().numpy().view(np.uint32), fe.cpu().numpy()
    for k, i in enumerate(idx.tolist()):
        if not 0 <= i < total:
            assert (ms[k], fe[k]) == (0xFFFFFFFF, 0xFF), i
            continue
        want = oracle.evaluate(scn, i)
        assert (int(ms[k]), int(fe[k])) == (want, int(want != 0xFFFFFFFF)), i
