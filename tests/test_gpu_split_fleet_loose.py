"""Fleets with much slack: calls that the band kernel leaves to the deque
kernel, by a sample of their loads, and scenarios that come back because a
deque outgrew its ring.  Costs, route counts and routes have the plain
kernel's bits on both sides of the line, whatever mixture of scenarios a call
holds, with several of them to a warp."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SAMPLE = 8  # scenarios that the choice looks at, the first and the last among them


def _cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _equal_to_plain(tour, Q, q, K, xy, flags=0):
    from paper_2602_05179_gb300 import api
    p = api.split_fleet_eval(tour, Q, q, K, coords=xy, algo="plain")
    api.status()
    r = api.split_fleet_eval(tour, Q, q, K, coords=xy)
    seen = api.status()
    assert seen & api.FLAG_DEVICE_CHECK == 0 and seen & flags == flags
    for key in ("cost", "nroutes", "route"):
        assert torch.equal(r[key], p[key]), key
    r = api.split_fleet_eval(tour, Q, q, K, coords=xy, routes=False)
    assert torch.equal(r["cost"], p["cost"]) and torch.equal(r["nroutes"], p["nroutes"])


def line(n, Q, K, S):
    """The sample's load from which on the band kernel keeps a call (0: always)."""
    idle = max(0.0, 1.0 - S / (24 * torch.cuda.get_device_properties(0).multi_processor_count))
    c = (27.0 + 6.0 * idle if K <= 32 else 43.0 + 3.0 * idle) + 1200.0 * idle / n - 49.0 * K / n
    m = max(K - c, min(3.0, K - c / 1.35))
    return int(SAMPLE * min(m, K + 1.0) * Q) if m >= 1 else 0


def _row(rng, n, Q, load):
    """Demands of at most Q that add up to `load` (at most n Q)."""
    w = rng.random(n) * (rng.random(n) < rng.uniform(0.3, 1.0)) + 1e-9
    q = np.minimum(np.floor(w / w.sum() * load), Q).astype(np.int64)
    for j in rng.permutation(n):  # the rest where there is room
        q[j] += max(min(load - int(q.sum()), Q - int(q[j])), 0)
    assert q.sum() == load
    return q


@pytest.mark.parametrize("n,K,S", [
    (5, 5, 300), (17, 16, 8000), (31, 24, 1000), (60, 24, 4000), (100, 24, 8000), (64, 32, 500),
    (64, 33, 500), (100, 64, 8000), (130, 40, 2000), (333, 32, 600), (200, 64, 1), (63, 60, 37),
])
@pytest.mark.parametrize("Q", [90, 300])
@pytest.mark.parametrize("above", [-1, 0])
def test_both_sides_of_the_line(n, K, S, Q, above):
    """A sample one below the line, and on it (with few positions it lies beyond
    what their demands can add up to: heavy rows then); all loads around it in
    the other scenarios, some with demands above Q and below 0."""
    rng = np.random.default_rng(n + K + Q)
    tour = _cuda((rng.permutation(n) + 1).astype(np.int32))
    xy = _cuda(rng.uniform(0, 100, (n + 1, 2)).astype(np.float32))
    q = np.zeros((S, n), np.int64)
    some = [_row(rng, n, Q, int(rng.integers(0, min(K, n) * Q + 1))) for _ in range(200)]
    for s in range(S):
        q[s] = some[s % 200]
    q[7::50, n // 2] = Q + 1
    q[9::50, 0] = -3
    sample = [(S - 1) * j // (SAMPLE - 1) for j in range(SAMPLE)]
    rows = sorted(set(sample))
    times = [sample.count(s) for s in rows]
    want = min(max(line(n, Q, K, S) + above, 0), SAMPLE * n * Q)
    assert S < 4000 or want > 0
    for s, c in zip(rows, times):  # each its share; the last ones, counted once, what is left
        q[s] = _row(rng, n, Q, min(want // SAMPLE, n * Q))
    left = want - sum(c * int(q[s].sum()) for s, c in zip(rows, times))
    for s, c in zip(rows, times):
        if c == 1 and left > 0:
            load = int(q[s].sum())
            q[s] = _row(rng, n, Q, min(load + left, n * Q))
            left -= int(q[s].sum()) - load
    assert left == 0 or S < SAMPLE or want // SAMPLE == n * Q
    _equal_to_plain(tour, Q, _cuda(q.astype(np.int32)), K, xy)


@pytest.mark.parametrize("n,K,S", [(60, 24, 9000), (100, 64, 20000), (200, 40, 1000)])
def test_outgrown_rings_come_back(n, K, S):
    """Customers at the depot: every candidate ties and stays in its deque."""
    from paper_2602_05179_gb300 import api
    rng = np.random.default_rng(n)
    tour = _cuda((rng.permutation(n) + 1).astype(np.int32))
    xy = rng.uniform(0, 100, (n + 1, 2)).astype(np.float32)
    xy[1:] = xy[0]
    for every in (1, 3, 40):  # all, a third, few outgrow; the others' windows are one or two long
        q = rng.integers(30, 60, (S, n)).astype(np.int32)
        q[::every] = rng.integers(0, 3, (len(q[::every]), n))
        if every > 1:  # the sample decides
            for j in range(SAMPLE):
                q[(S - 1) * j // (SAMPLE - 1)] = rng.integers(0, 3, n)
        _equal_to_plain(tour, 90, _cuda(q), K, _cuda(xy), api.FLAG_FALLBACK)
