"""The FP64 scenario mean (one launch; eight values at a time as a float pair)
against numpy's FP64 sum of the returned costs, at the edges of its groups,
blocks and grids, and with infinite costs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [1, 255, 2047, 2048, 2049, 4096, 4097, 100_003, 1_048_576, 1_100_000])
def test_mean_is_the_fp64_mean(S):
    from paper_2602_05179_gb300 import api
    rng = np.random.default_rng(S)
    T = 2  # values spread over six decades: h, p and f scale the costs
    cons = torch.from_numpy(rng.integers(0, 1000, (S, T)).astype(np.int32)).cuda()
    fixed = torch.from_numpy(np.array([1e-3, 1e3], np.float32)).cuda()
    r = api.reinsert_eval(T, 30, 7, 1e-3, 3.7, 0.0, fixed, cons)
    v = r["value"].cpu().numpy().astype(np.float64)
    assert abs(float(r["mean"]) - v.mean()) <= 1e-14 * np.abs(v).sum() / S
    again = api.reinsert_eval(T, 30, 7, 1e-3, 3.7, 0.0, fixed, cons)
    assert float(again["mean"]) == float(r["mean"])


def test_mean_with_infeasible_scenarios():
    from paper_2602_05179_gb300 import api
    rng = np.random.default_rng(1)
    n, S = 20, 10_000
    tour = torch.from_numpy((rng.permutation(n) + 1).astype(np.int32)).cuda()
    xy = torch.from_numpy(rng.uniform(0, 100, (n + 1, 2)).astype(np.float32)).cuda()
    q = torch.from_numpy(rng.integers(1, 11, (S, n)).astype(np.int32)).cuda()
    assert torch.isfinite(api.split_eval(tour, 10, q, coords=xy)["mean"])
    q[1234, 5] = 11
    assert float(api.split_eval(tour, 10, q, coords=xy)["mean"]) == float("inf")
    api.status()
