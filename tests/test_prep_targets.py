"""Candidates of prediction targets (one grid of the training points, queries dealt over threads) against a full sort:
no targets, fewer training points than candidates, ties and coincident points, counts around the queries' chunks."""
import numpy as np
import pytest

import synthetic
from paper_2307_11648_gb300 import sic


@pytest.mark.parametrize("n,nt,C,dim,threads", [(40, 0, 8, 2, 0), (40, 39, 8, 3, 2), (300, 7, 400, 1, 1),
                                                (900, 8, 33, 2, 3), (900, 9, 128, 3, 0), (2000, 250, 64, 2, 4)])
@pytest.mark.parametrize("ties", [False, True])
def test_against_a_full_sort(n, nt, C, dim, threads, ties):
    p = synthetic.points(n, dim, 4)
    if ties:
        p = np.round(6 * p) / 6
    ptr, idx = sic.prep_candidates_targets(p, nt, C, threads)
    assert ptr[0] == 0 and len(idx) == ptr[-1]
    for t in range(nt):
        d = np.zeros(n - nt)
        for c in range(dim):
            d += (p[nt:, c] - p[t, c]) ** 2
        want = nt + np.lexsort((np.arange(n - nt), d))[:C]
        assert np.array_equal(idx[ptr[t]:ptr[t + 1]], want)
