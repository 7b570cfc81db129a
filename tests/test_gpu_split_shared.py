"""The shared-demand kernel of batched plans (one length, one demand array)
gives the bits of the single-tour Split: tours that fill and do not fill
record blocks, ragged last tiles, both staging types, demands above Q and
below 0, flagged scenarios."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("case", [
    # n, S, B, Q, demand range, ties
    (1, 40, 64, 30, (1, 20), False),
    (15, 33, 64, 30, (1, 20), False),
    (16, 64, 65, 30, (1, 20), False),
    (17, 31, 70, 400, (1, 60), False),       # 16-bit staging
    (33, 1000, 64, 60, (1, 20), False),
    (100, 5000, 67, 100, (1, 30), False),    # several tiles per CTA and CTAs per tile
    (48, 100, 64, 20, (-2, 22), False),      # demands above Q and below 0
    (64, 70, 64, 60, (0, 3), True),          # zero costs: windows above the ring are recomputed
])
def test_shared_equals_single(case):
    from paper_2602_05179_gb300 import api
    n, S, B, Q, (lo, hi), ties = case
    rng = np.random.default_rng(n + S)
    xy = rng.uniform(0, 100, (n + 1, 2)).astype(np.float32)
    if ties:
        xy[:] = 50.0
    tours = np.stack([rng.permutation(n) + 1 for _ in range(B)]).astype(np.int32)
    q = _cuda(rng.integers(lo, hi + 1, (S, n)).astype(np.int32))
    t, c = _cuda(tours.reshape(-1)), _cuda(np.tile(xy, (B, 1)))
    plan = api.SplitPlan([n] * B, t, c, q, Q, S, dem_off=[0] * B)
    costs, means = plan.run()
    assert plan.info()["warps_per_cta"] == -2
    flags = api.status()
    assert bool(flags & api.FLAG_FALLBACK) == ties and flags & api.FLAG_DEVICE_CHECK == 0
    for b in range(B):
        r = api.split_eval(_cuda(tours[b]), Q, q, coords=_cuda(xy), algo="plain")
        assert torch.equal(costs[b], r["cost"]), b
    plan.close()
