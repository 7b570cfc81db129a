"""Horizons at which the reachable-state kernel (AUTO) leaves calls of little
consumption to the lane kernel: values, policies and means are the warp
kernel's bits on both sides of the line and in calls that mix scenarios."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SAMPLE = 8  # scenarios that the choice looks at, the first and the last among them


def line(T, U, K, table):
    """The sample's consumption from which on the chains keep a call."""
    states = 32 * ((U + 32) // 32)
    t0 = 16 + states / 2 if K > 4 else 32 + 0.75 * states if K else 1.25 * states
    assert states >= 64 and (table or K) and T > t0
    cells = (T / 2 + 20) / (T / t0) ** 1.5 - 20
    days = T * (1 - math.sqrt(max(0.0, 1 - 2 * cells / T)))
    return int(SAMPLE * T * U / max(days, 1.0))


@pytest.mark.parametrize("T,U,K,table,S", [
    (90, 40, 0, True, 300), (128, 63, 0, True, 2000), (121, 95, 0, True, 65),
    (85, 50, 1, False, 300), (99, 63, 4, False, 33), (49, 40, 5, False, 300),
    (80, 63, 8, False, 2000), (80, 80, 6, False, 1), (65, 64, 7, False, 9),
])
@pytest.mark.parametrize("above", [-1, 0])
def test_both_sides_of_the_line(T, U, K, table, S, above):
    from paper_2602_05179_gb300 import api
    rng = np.random.default_rng(T + U + K)
    cons = rng.poisson(rng.choice([0.05, 2.0, 9.0, 70.0], (S, 1)), (S, T)).astype(np.int32)
    cons[3::50, T // 2] = 1 << 20  # far above U: counts as U
    want = line(T, U, K, table) + above
    sample = [(S - 1) * j // (SAMPLE - 1) for j in range(SAMPLE)]
    rows = sorted(set(sample))
    left = want
    for n, s in enumerate(rows):  # an equal share each, the last row what is left
        share = left if s == rows[-1] and sample.count(s) == 1 else want // SAMPLE
        cons[s] = share // T
        cons[s, : share % T] += 1
        assert cons[s].max() <= U
        left -= share * sample.count(s)
    assert left == 0 or S < SAMPLE
    cons = torch.from_numpy(cons).cuda()
    fixed = torch.from_numpy(rng.uniform(5, 50, T).astype(np.float32)).cuda()
    kw = {}
    if table:
        kw["table"] = torch.from_numpy(rng.uniform(0, 30, U + 1).astype(np.float32)).cuda()
    if K:
        kw["route_cost"] = torch.from_numpy(rng.uniform(5, 50, (T, K)).astype(np.float32)).cuda()
        kw["route_cap"] = torch.from_numpy(rng.integers(0, int(1.25 * U), (S, T, K)).astype(np.int32)).cuda()
    args = (T, U, U // 2, 1.25, 20.0, 0.25, None if K else fixed, cons)
    ref = api.reinsert_eval(*args, algo="warp", **kw)
    for out in ({}, {"policy": False}, {"mean": False}, {"policy": False, "mean": False}):
        r = api.reinsert_eval(*args, **kw, **out)
        for key in ("value", "policy", "mean"):
            assert r[key] is None if out.get(key) is False else torch.equal(r[key], ref[key]), key
