"""When SplitMeanCost's forward counts the routes as it evaluates: for tours up to
64, and up to 42 tiles per SM; beyond, the forward is the evaluation alone.
Mean and gradient are the same bits on both sides of each line."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,Q,tiles,over,fused", [
    (64, 100, 60, 0, True),
    (65, 100, 42, 0, True),
    (65, 100, 42, 1, False),
    (120, 300, 42, 0, True),
    (120, 300, 42, 1, False),
    (200, 300, 20, 0, True),      # one round of 20 warps, and a second one begun
    (200, 300, 20, 1, True),
    (336, 100, 24, 1, True),
    (500, 100, 42, 0, True),
    (500, 100, 42, 1, False),
    (513, 100, 1, 0, False),      # rows that the kernel does not hold
])
def test_choice_and_bits(n, Q, tiles, over, fused):
    from paper_2602_05179_gb300 import api
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    S = 32 * tiles * sms + over
    rng = np.random.default_rng(n + Q)
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    xy = torch.from_numpy(rng.uniform(0, 100, (n + 1, 2))).cuda()
    dist = (xy[:, None] - xy[None]).square().sum(-1).sqrt().float().contiguous()
    tour = torch.from_numpy((rng.permutation(n) + 1).astype(np.int32)).cuda()
    q = torch.randint(1, 20, (S, n), generator=g, dtype=torch.int32, device="cuda")
    assert (api._split_mean_routes(tour, Q, q, dist)[1] is not None) == fused
    leaf = dist.clone().requires_grad_(True)
    mean = api.SplitMeanCost.apply(leaf, tour, q, Q)
    mean.backward()
    ref = api.split_eval(tour, Q, q, dist=dist)["mean"]
    grad, _ = api.split_backward(tour, Q, q, dist, torch.ones((), device="cuda"))
    assert torch.equal(mean.detach().view(torch.int64), ref.view(torch.int64))
    assert torch.equal(leaf.grad, grad)
