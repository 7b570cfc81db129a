"""How split_shared.cu deals the (tile, tour) pairs of small launches: CTAs of
one tile each, or runs that cross tiles.  Every cost is written once and has
the plain kernel's bits, on both sides of the choice."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("B,S", [(64, 1), (64, 32), (65, 500), (100, 500), (70, 2000), (100, 2560),
                                 (126, 2464), (64, 4800), (64, 4865), (200, 1535), (1025, 32)])
def test_every_pair_once(B, S):
    from paper_2602_05179_gb300 import api
    n, Q = 21, 60
    rng = np.random.default_rng(B + S)
    xy = rng.uniform(0, 100, (n + 1, 2)).astype(np.float32)
    base = rng.permutation(n) + 1
    tours = np.stack([np.concatenate([base[:k], rng.permutation(base[k:])])
                      for k in rng.integers(0, n, B)]).astype(np.int32)
    q = _cuda(rng.integers(1, 20, (S, n)).astype(np.int32))
    plan = api.SplitPlan([n] * B, _cuda(tours.reshape(-1)), _cuda(np.tile(xy, (B, 1))), q, Q, S, dem_off=[0] * B)
    plan.costs.fill_(-1.0)
    costs, means = plan.run()
    assert plan.info()["warps_per_cta"] == -2
    for b in range(B) if B <= 200 else rng.choice(B, 150, replace=False):
        r = api.split_eval(_cuda(tours[b]), Q, q, coords=_cuda(xy), algo="plain")
        assert torch.equal(costs[b], r["cost"]), b
    assert bool((costs > 0).all())
    plan.close()
