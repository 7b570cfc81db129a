"""Forms in which a gradient and the saved tensors reach SplitMeanCost's
backward, which hands their memory to the kernels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _problem(n=40, S=90, Q=50, seed=4):
    rng = np.random.default_rng(seed)
    tour = torch.from_numpy((rng.permutation(n) + 1).astype(np.int32)).cuda()
    qd = torch.from_numpy(rng.integers(1, 9, (S, n)).astype(np.int32)).cuda()
    leaf = torch.from_numpy(rng.uniform(1, 9, (n + 1, n + 1)).astype(np.float32)).cuda().requires_grad_(True)
    return leaf, tour, qd, Q


@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
def test_lazily_negated_gradient(dt):
    """A real tensor can carry its negation as a flag; the sign counts."""
    from paper_2602_05179_gb300 import api
    leaf, tour, qd, Q = _problem()
    m = api.SplitMeanCost.apply(leaf, tour, qd, Q)
    g, = torch.autograd.grad(m, leaf, retain_graph=True)
    neg = torch._neg_view(torch.ones((), dtype=torch.float64, device="cuda"))
    assert neg.is_neg() and float(neg) == -1.0
    if dt == torch.float64:
        gn, = torch.autograd.grad(m, leaf, neg)
    else:  # as backward sees a float gradient
        gn = api._grad_from_routes(tour, qd.shape[0], api._split_mean_routes(tour, Q, qd, leaf.detach())[1],
                                   torch._neg_view(torch.ones((), dtype=dt, device="cuda")))
    assert torch.equal(gn, -g)


@pytest.mark.parametrize("form", ["int64", "strided"])
@pytest.mark.parametrize("which", ["tour", "routes"])
def test_unpacked_tensors_of_another_form_are_refused(which, form):
    """A saved-tensor hook's unpacked tour or route counts are checked as the
    forward's inputs are."""
    from paper_2602_05179_gb300 import api
    leaf, tour, qd, Q = _problem()
    n = tour.numel()

    def unpack(t):
        hit = t.dtype == torch.int32 and t.numel() == n if which == "tour" else t.numel() == 2 * n + 1
        if not hit:
            return t
        if form == "int64":
            return t.to(torch.int64 if which == "tour" else torch.int32)
        return torch.stack((t, t), 1)[:, 0]

    with torch.autograd.graph.saved_tensors_hooks(lambda t: t, unpack):
        m = api.SplitMeanCost.apply(leaf, tour, qd, Q)
        with pytest.raises(ValueError):
            m.backward()
