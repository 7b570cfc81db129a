"""Tours resumed from tour 0's kept states in bulk: each CTA has hundreds of
tours on a tile, so nearly all are claimed when the states exist.  8- and
16-bit staging, states 8 and more positions apart, lanes whose deque outgrew
its ring before the state they resume from (customers on a ray: each candidate
is worse than the one before, so a restarted deque gives a higher cost unless
the scenario is recomputed).  Costs have the plain kernel's bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("n,S,B,Q,hi,ray", [
    (24, 4864, 2000, 60, 20, False),
    (100, 2432, 1024, 100, 20, False),
    (100, 2432, 1024, 400, 60, False),     # 16-bit staging
    (600, 1280, 1024, 400, 30, False),     # states more than 8 positions apart
    (120, 1280, 1024, 90, 8, True),        # windows of 20: rings outgrow in the first half
    (200, 1280, 1024, 700, 60, True),
])
def test_bulk_resume(n, S, B, Q, hi, ray):
    from paper_2602_05179_gb300 import api
    rng = np.random.default_rng(n + B)
    xy = rng.uniform(0, 100, (n + 1, 2)).astype(np.float32)
    tour0 = rng.permutation(n) + 1
    if ray:
        xy[0] = 0.0
        xy[tour0[: n // 2]] = np.stack([np.arange(1, n // 2 + 1) / 4.0, np.zeros(n // 2)], 1)
    tours = []
    for b in range(B):
        t = tour0.copy()
        i, j = sorted(rng.integers(n // 8, n, 2)) if b else (0, 0)
        t[i:j + 1] = t[i:j + 1][::-1]
        tours.append(t)
    tours = np.stack(tours).astype(np.int32)
    q = _cuda(rng.integers(1, hi + 1, (S, n)).astype(np.int32))
    plan = api.SplitPlan([n] * B, _cuda(tours.reshape(-1)), _cuda(np.tile(xy, (B, 1))), q, Q, S, dem_off=[0] * B)
    api.status()
    costs, _ = plan.run()
    assert plan.info()["warps_per_cta"] == -2
    assert bool(api.status() & api.FLAG_FALLBACK) or not ray
    tours, xy = _cuda(tours), _cuda(xy)
    for b in range(B):
        r = api.split_eval(tours[b], Q, q, coords=xy, algo="plain", mean=False)
        assert torch.equal(costs[b], r["cost"]), b
    plan.close()
