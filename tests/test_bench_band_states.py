"""The states that bench.py credits the fleet-limited Split with, by brute force:
(k, i), i >= 1, where some way of at most k routes leads from the start to i and
some way of at most K - k from i to the end."""
import numpy as np
import pytest

import bench


def _reached(row, Q, start, routes):
    """Positions that at most `routes` routes reach from `start`."""
    seen = {start}
    for _ in range(routes):
        seen |= {j for i in seen for j in range(i + 1, len(row) + 1) if row[i:j].sum() <= Q}
    return seen


@pytest.mark.parametrize("n,Q,K,hi", [(1, 5, 1, 5), (6, 10, 3, 6), (7, 9, 7, 9), (8, 12, 4, 7), (8, 12, 3, 13)])
def test_band_states_by_brute_force(n, Q, K, hi):
    rng = np.random.default_rng(n + K)
    tour = rng.permutation(n) + 1
    q = rng.integers(0, hi + 1, (40, n))
    got = bench.band_states(q, tour, Q, K)
    for s, row in enumerate(q[:, tour - 1]):
        want = 0
        if n in _reached(row, Q, 0, K):
            want = sum(i > 0 and n in _reached(row, Q, i, K - k)
                       for k in range(1, K + 1) for i in _reached(row, Q, 0, k))
        assert got[s] == want, s
