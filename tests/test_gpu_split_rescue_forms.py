"""The recomputation of flagged scenarios (split_rescue.cu) with soft capacity
and with route counts: the plain kernel's bits, at block edges of 32
positions, for penalties that let few or all earlier positions compete."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _case(n, seed):
    rng = np.random.default_rng(seed)
    xy = rng.uniform(0, 100, (n + 1, 2)).astype(np.float32)
    return rng, _cuda((rng.permutation(n) + 1).astype(np.int32)), xy


@pytest.mark.parametrize("beta", [0.0, 0.01, 3.0, 500.0])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 65, 200])
def test_soft_rescue_equals_plain(n, beta):
    from paper_2602_05179_gb300 import api
    rng, tour, xy = _case(n, n)
    S, Q = 40, 100
    q = rng.integers(0, 30, (S, n)).astype(np.int32)
    q[np.arange(S), rng.integers(0, n, S)] = 300  # beyond the 8-bit staging: every scenario is flagged
    args = (tour, Q, _cuda(q))
    for preds in ("u16", "i32", None):
        kw = dict(coords=_cuda(xy), overload_penalty=beta, preds=preds)
        r = api.split_eval(*args, **kw)
        assert api.status() & api.FLAG_FALLBACK
        p = api.split_eval(*args, algo="plain", **kw)
        assert torch.equal(r["cost"], p["cost"])
        assert preds is None or torch.equal(r["pred"], p["pred"])


def test_soft_rescue_loads_beyond_31_bits():
    """Route loads that wrap, as the plain kernel's do."""
    from paper_2602_05179_gb300 import api
    rng, tour, xy = _case(70, 5)
    q = rng.integers(2**29, 2**30, (33, 70)).astype(np.int32)
    kw = dict(coords=_cuda(xy), overload_penalty=1e-6, preds="i32")
    r = api.split_eval(tour, 100, _cuda(q), **kw)
    p = api.split_eval(tour, 100, _cuda(q), algo="plain", **kw)
    assert torch.equal(r["cost"], p["cost"]) and torch.equal(r["pred"], p["pred"])


@pytest.mark.parametrize("n", [33, 64, 150])
def test_route_counts_of_flagged_scenarios(n):
    """Travel costs of zero: every candidate ties, windows of more than a
    ring's entries flag every scenario, and the counts are the plain kernel's."""
    from paper_2602_05179_gb300 import api
    rng, tour, _ = _case(n, n + 1)
    S, Q = 70, 60
    q = rng.integers(0, 4, (S, n)).astype(np.int32)
    q[3, n // 2] = 61  # one infeasible scenario: not counted
    dist = torch.zeros((n + 1, n + 1), device="cuda")
    one = torch.ones((), device="cuda")
    api.status()
    g, h = api.split_backward(tour, Q, _cuda(q), dist, one, want_hist=True)
    assert api.status() & api.FLAG_FALLBACK
    gp, hp = api.split_backward(tour, Q, _cuda(q), dist, one, want_hist=True, algo="plain")
    assert torch.equal(h, hp) and torch.equal(g, gp)
