"""When SplitMeanCost's forward counts the routes as it evaluates: in one round
of the adjoint's kernel, where that costs a forward without a backward nothing,
and for short tours; beyond, the forward is the evaluation alone.  Mean and
gradient are the same bits on both sides of each line."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _round(n, Q):
    """Scenarios of one round: as many warps per SM, 16 to 24, as have tensor
    memory columns for a row (rows take a multiple of four)."""
    words = ((n if Q <= 254 else 2 * n) + 15) // 16 * 4
    warps = max(w for w in range(16, 25) if words <= (512 // ((w + 3) // 4) & ~3))
    return 32 * warps * torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("n,Q,over,fused", [
    (50, 100, 40_000, True),
    (51, 100, 0, True),
    (51, 100, 1, False),
    (100, 300, 0, True),
    (100, 300, 1, False),
    (200, 300, 0, True),      # rows of 400 bytes: 20 warps
    (200, 300, 1, False),
    (336, 100, 0, True),
    (336, 100, 1, False),
    (337, 100, -50_000, False),
])
def test_choice_and_bits(n, Q, over, fused):
    from paper_2602_05179_gb300 import api
    S = _round(n, Q) + over
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
