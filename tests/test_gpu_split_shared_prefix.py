"""Tours that begin as tour 0 does are resumed from its kept states
(split_shared.cu): every shared length around the kept positions, tours equal
to tour 0, records that differ only in a coordinate, flagged and infeasible
scenarios, lengths whose states are more than 8 positions apart."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("case", [
    # n, S, B, Q, demand range, ties
    (9, 40, 64, 30, (1, 20), False),
    (24, 64, 64, 300, (1, 60), False),
    (100, 700, 240, 100, (1, 30), False),
    (100, 64, 240, 20, (-2, 22), False),
    (67, 70, 96, 60, (0, 3), True),
    (600, 100, 70, 400, (1, 30), False),
    (127, 40, 64, 100, (1, 30), False),      # states that fill the shared memory to within 16 bytes
    (64, 40, 64, 300, (1, 60), False),
])
def test_prefixes_equal_single(case):
    from paper_2602_05179_gb300 import api
    n, S, B, Q, (lo, hi), ties = case
    rng = np.random.default_rng(3 * n + S)
    xy = rng.uniform(0, 100, (n + 1, 2)).astype(np.float32)
    if ties:
        xy[:] = 50.0
    tour0 = rng.permutation(n) + 1
    tours, coords = [], []
    for b in range(B):
        t, c = tour0.copy(), xy.copy()
        keep = (b * 37) % (n + 1) if b else n
        t[keep:] = rng.permutation(t[keep:])
        if b % 5 == 4:  # the same tour, one customer elsewhere
            t = tour0.copy()
            c[t[min(keep, n - 1)]] += 1.0
        tours.append(t)
        coords.append(c)
    tours, coords = np.stack(tours).astype(np.int32), np.stack(coords)
    q = _cuda(rng.integers(lo, hi + 1, (S, n)).astype(np.int32))
    plan = api.SplitPlan([n] * B, _cuda(tours.reshape(-1)), _cuda(coords.reshape(-1, 2)), q, Q, S, dem_off=[0] * B)
    for _ in range(2):
        costs, _ = plan.run()
        assert plan.info()["warps_per_cta"] == -2
        for b in range(B):
            r = api.split_eval(_cuda(tours[b]), Q, q, coords=_cuda(coords[b]), algo="plain")
            assert torch.equal(costs[b], r["cost"]), b
    plan.close()
