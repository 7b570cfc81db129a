"""The band kernel of the fleet-limited Split (AUTO) against the plain kernel,
bit for bit: costs, route counts and routes, where the band is narrow, the
whole tour or empty, and on both sides of the window length that sends a
scenario to the wide form."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("case", [
    # n, S, Q, demand range, K, ties
    (31, 40, 30, (1, 15), 14, False),     # odd rows, about one route of slack
    (64, 97, 60, (1, 20), 13, False),     # some scenarios infeasible
    (96, 64, 60, (1, 20), 64, False),     # no binding limit: the band is the tour
    (100, 64, 320, (9, 11), 5, False),    # windows of 29 to 35: both forms
    (200, 33, 400, (0, 6), 8, False),     # wide windows, zero demands
    (128, 50, 12, (4, 12), 60, False),    # windows of one to three positions
    (130, 50, 10, (8, 12), 64, False),    # demands above Q
    (61, 40, 60, (1, 20), 14, True),      # exact ties
    (700, 24, 200, (1, 30), 60, False),
])
def test_band_equals_plain(case):
    from paper_2602_05179_gb300 import api
    n, S, Q, (lo, hi), K, ties = case
    rng = np.random.default_rng(n + K)
    tour = _cuda((rng.permutation(n) + 1).astype(np.int32))
    xy = rng.uniform(0, 100, (n + 1, 2)).astype(np.float32)
    if ties:  # customers on a ray from the depot, at whole distances
        xy[:] = 0.0
        xy[1:, 0] = rng.integers(1, 5, n)
    q = _cuda(rng.integers(lo, hi + 1, (S, n)).astype(np.int32))
    xy = _cuda(xy)
    p = api.split_fleet_eval(tour, Q, q, K, coords=xy, algo="plain")
    off = torch.empty(S * n + 1, dtype=torch.int32, device="cuda")[1:].view(S, n).copy_(q)
    for dem in (q, off):  # rows on and off 16 bytes
        r = api.split_fleet_eval(tour, Q, dem, K, coords=xy)
        for key in ("cost", "nroutes", "route"):
            assert torch.equal(r[key], p[key]), key
    r = api.split_fleet_eval(tour, Q, q, K, coords=xy, routes=False)
    assert torch.equal(r["cost"], p["cost"]) and torch.equal(r["nroutes"], p["nroutes"])
    assert api.status() & api.FLAG_DEVICE_CHECK == 0
