"""The fleet-limited Split's other paths against the plain kernel, bit for bit:
the band kernel with several scenarios to a warp (its rows, offsets and lists
used again), and the deque kernel with its own recomputation, which AUTO takes
for tours whose rows do not fit the band kernel's shared memory."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _equal(tour, Q, q, K, xy):
    from paper_2602_05179_gb300 import api
    p = api.split_fleet_eval(tour, Q, q, K, coords=xy, algo="plain")
    api.status()
    r = api.split_fleet_eval(tour, Q, q, K, coords=xy)
    flags = api.status()
    assert flags & api.FLAG_DEVICE_CHECK == 0
    for key in ("cost", "nroutes", "route"):
        assert torch.equal(r[key], p[key]), key
    r = api.split_fleet_eval(tour, Q, q, K, coords=xy, routes=False)
    assert torch.equal(r["cost"], p["cost"]) and torch.equal(r["nroutes"], p["nroutes"])
    return flags, p


@pytest.mark.parametrize("n,K,Q", [(31, 8, 90), (64, 13, 100), (100, 12, 150), (99, 12, 400)])
def test_band_with_several_scenarios_to_a_warp(n, K, Q):
    """Narrow, wide and infeasible scenarios mixed, three or more to a warp."""
    from paper_2602_05179_gb300 import api
    S = 3 * 24 * torch.cuda.get_device_properties(0).multi_processor_count + 5
    rng = np.random.default_rng(n)
    tour = _cuda((rng.permutation(n) + 1).astype(np.int32))
    xy = _cuda(rng.uniform(0, 100, (n + 1, 2)).astype(np.float32))
    hi = max(2, int(1.7 * K * Q / n))
    q = rng.integers(1, min(hi, Q) + 1, (S, n))
    q[1::3] = rng.integers(0, 3, q[1::3].shape)                       # windows above 32
    q[1::3, tour.cpu().numpy()[: n // 3] - 1] = min(hi, Q)            # behind short ones
    q[4::31, n // 2] = Q + 1
    flags, p = _equal(tour, Q, _cuda(q.astype(np.int32)), K, xy)
    assert flags & api.FLAG_INFEASIBLE and torch.isfinite(p["cost"]).float().mean() > 0.2
    assert bool(flags & api.FLAG_FALLBACK) == (n > 32)


@pytest.mark.parametrize("n,K,Q,ties", [
    (1900, 24, 1200, False), (2000, 33, 1000, False), (1951, 64, 500, False),
    (1900, 20, 1500, True), (2000, 40, 900, True),
])
def test_long_tours_take_the_deque_kernel(n, K, Q, ties):
    """Above the band's longest tour; with ties (customers at the depot) every
    window outgrows the ring and is recomputed."""
    from paper_2602_05179_gb300 import api
    S = 40
    rng = np.random.default_rng(n + K)
    tour = _cuda((rng.permutation(n) + 1).astype(np.int32))
    xy = rng.uniform(0, 100, (n + 1, 2)).astype(np.float32)
    if ties:
        xy[1:] = xy[0]
    mean = K * Q / n / 1.1
    q = rng.integers(1, int(2 * mean), (S, n)).astype(np.int32)
    q[3, n // 2] = Q + 1
    flags, p = _equal(tour, Q, _cuda(q), K, _cuda(xy))
    assert flags & api.FLAG_INFEASIBLE and torch.isfinite(p["cost"]).float().mean() > 0.5
    if ties:
        assert flags & api.FLAG_FALLBACK
