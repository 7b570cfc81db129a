"""SplitMeanCost's single pass (costs and route counts from one kernel)
against split_eval and split_backward: the same mean and gradient bits, at
tile edges, with infeasible, flagged (zero travel costs: every candidate
ties) and unreachable customers, and for fp32 and fp64 upstream gradients."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("kind", ["plain", "infeasible", "flagged", "unreachable"])
@pytest.mark.parametrize("n,S,Q", [(1, 1, 40), (3, 31, 40), (33, 33, 60), (150, 5000, 100),
                                   (256, 700, 300), (512, 65, 120), (513, 70, 120)])
def test_mean_and_gradient_bits(n, S, Q, kind):
    from paper_2602_05179_gb300 import api
    rng = np.random.default_rng(n + S)
    xy = rng.uniform(0, 100, (n + 1, 2))
    dist = np.hypot(*(xy[:, None] - xy[None]).transpose(2, 0, 1)).astype(np.float32)
    q = rng.integers(0 if kind == "flagged" else 1, 4 if kind == "flagged" else 30, (S, n)).astype(np.int32)
    if kind == "infeasible":
        q[::3, n // 2] = Q + 1
    if kind == "flagged":
        dist[:] = 0.0
    if kind == "unreachable":
        dist[0, n // 3 + 1] = dist[n // 2 + 1, 0] = np.inf
    tour, qd, d = _cuda((rng.permutation(n) + 1).astype(np.int32)), _cuda(q), _cuda(dist)
    ref = api.split_eval(tour, Q, qd, dist=d)["mean"]
    for scale, dt in ((1.0, torch.float64), (0.1, torch.float32)):
        leaf = d.clone().requires_grad_(True)
        mean = api.SplitMeanCost.apply(leaf, tour, qd, Q)
        assert torch.equal(mean.detach().view(torch.int64), ref.view(torch.int64))
        (mean.to(dt) * scale).backward()
        gm = torch.tensor(scale, dtype=dt, device="cuda")
        g, _ = api.split_backward(tour, Q, qd, d, gm)
        assert torch.equal(leaf.grad, g)
        with torch.no_grad():
            m = api.SplitMeanCost.apply(leaf, tour, qd, Q)
        assert not m.requires_grad and torch.equal(m.view(torch.int64), ref.view(torch.int64))


def test_saved_inputs_and_second_backward():
    """A changed input is still refused, and the counts serve two backwards."""
    from paper_2602_05179_gb300 import api
    rng = np.random.default_rng(4)
    tour = _cuda((rng.permutation(40) + 1).astype(np.int32))
    qd = _cuda(rng.integers(1, 9, (90, 40)).astype(np.int32))
    leaf = torch.rand((41, 41), device="cuda", requires_grad=True)
    m = api.SplitMeanCost.apply(leaf, tour, qd, 50)
    g1, = torch.autograd.grad(m, leaf, retain_graph=True)
    g2, = torch.autograd.grad(m, leaf, retain_graph=True)
    assert torch.equal(g1, g2)
    qd.add_(1)
    with pytest.raises(RuntimeError):
        m.backward()
