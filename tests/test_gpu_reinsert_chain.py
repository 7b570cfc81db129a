"""The reachable-state kernel (AUTO without the C_0 table) gives the bits of
the kernels that evaluate every state: values, policies and means, over the
shapes and inputs where its chains start, end or stay empty."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [
    # T, U, I0, S, consumption, unit cost, table, cost range
    (1, 50, 50, 37, ("poisson", 20.0), 0.0, False, (5, 50)),      # one day, full stock
    (2, 8, 0, 33, ("poisson", 3.0), 0.5, False, (5, 50)),         # one pair of chains, empty stock
    (13, 40, 17, 65, ("poisson", 6.0), 0.0, False, (5, 50)),      # odd T: day 0 alone, rows of 13 bytes
    (60, 200, 100, 1000, ("poisson", 8.0), 0.0, False, (5, 50)),  # the workload's shape, a last tile of 8
    (60, 0, 0, 33, ("poisson", 3.0), 0.0, False, (5, 50)),        # no stock at all
    (28, 31, 31, 70, ("poisson", 40.0), 0.25, False, (5, 50)),    # every day sells out
    (40, 63, 63, 96, ("zeros", 0.9), 0.0, False, (5, 50)),        # days without consumption: chains of T days
    (41, 63, 63, 96, ("zeros", 0.7), 0.0, False, (-20, 20)),      # ... with costs below zero at a full stock
    (24, 20, 20, 64, ("zeros", 0.5), -0.5, False, (-5, 30)),
    (36, 100, 50, 90, ("huge", 0.1), 0.5, False, (5, 50)),        # consumption far above U
    (30, 70, 3, 50, ("poisson", 9.0), 0.4, True, (5, 50)),        # table end costs
    (20, 255, 9, 40, ("poisson", 40.0), 0.0, True, (5, 50)),
    (32, 300, 17, 40, ("poisson", 30.0), 0.2, False, (5, 50)),    # U above 255
    (126, 200, 200, 64, ("poisson", 8.0), 0.0, False, (5, 50)),   # near the longest horizon
]


def _cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _consumption(rng, S, T, U, kind):
    what, v = kind
    if what == "zeros":
        return rng.poisson(5.0, (S, T)) * (rng.random((S, T)) > v)
    if what == "huge":
        d = rng.poisson(8.0, (S, T)).astype(np.int64)
        far = rng.random((S, T)) < v
        d[far] = rng.integers(U, 2**31 - 1, far.sum())
        return d
    return rng.poisson(v, (S, T))


def _same(a, b):
    for key in ("value", "policy", "mean"):
        assert torch.equal(a[key], b[key]), key


@pytest.mark.parametrize("case", CASES)
def test_chain_equals_all_states(case):
    from paper_2602_05179_gb300 import api
    T, U, I0, S, kind, c, use_table, (flo, fhi) = case
    rng = np.random.default_rng(T * 1000 + U)
    cons = _cuda(_consumption(rng, S, T, U, kind).astype(np.int32))
    fixed = _cuda(rng.uniform(flo, fhi, T).astype(np.float32))
    table = _cuda(rng.uniform(0, 30, U + 1).astype(np.float32)) if use_table else None
    args = (T, U, I0, 1.25, 20.0, c, fixed, cons)
    ref = api.reinsert_eval(*args, table=table, algo="warp")
    _same(api.reinsert_eval(*args, table=table), ref)
    # rows and outputs off 16 bytes: the scalar loads and stores
    off = torch.empty(S * T + 1, dtype=torch.int32, device="cuda")[1:].view(S, T).copy_(cons)
    _same(api.reinsert_eval(T, U, I0, 1.25, 20.0, c, fixed, off, table=table), ref)


@pytest.mark.parametrize("K", [1, 3, 4, 5, 8])
@pytest.mark.parametrize("case", [
    (13, 40, 17, 65, ("poisson", 6.0), 0.5, (5, 50)),
    (60, 200, 100, 500, ("poisson", 8.0), 0.0, (5, 50)),
    (40, 63, 63, 96, ("zeros", 0.8), 0.0, (-20, 20)),
    (24, 255, 255, 64, ("huge", 0.1), 0.25, (5, 50)),
])
def test_chain_routes_equal_all_states(case, K):
    from paper_2602_05179_gb300 import api
    T, U, I0, S, kind, c, (flo, fhi) = case
    rng = np.random.default_rng(T * 1000 + U + K)
    cons = _cuda(_consumption(rng, S, T, U, kind).astype(np.int32))
    rcost = rng.uniform(flo, fhi, (T, K)).astype(np.float32)
    if K > 2:
        rcost[:, 2] = rcost[:, 0]  # ties go to the first route
    cap = rng.integers(-3, int(1.25 * U) + 2, (S, T, K)).astype(np.int32)
    kw = dict(route_cost=_cuda(rcost), route_cap=_cuda(cap))
    ref = api.reinsert_eval(T, U, I0, 1.25, 20.0, c, None, cons, algo="warp", **kw)
    _same(api.reinsert_eval(T, U, I0, 1.25, 20.0, c, None, cons, **kw), ref)
