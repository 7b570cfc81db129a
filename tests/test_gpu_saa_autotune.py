"""The search's autotuner times its plan on tours that the search scores."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_autotune_runs_the_first_iterations_tours():
    """Before any iteration the plan is timed on the first one's neighbours: the
    means it leaves are those that the iteration then finds.  After one, its
    tours are kept."""
    from paper_2602_05179_gb300 import api
    rng = np.random.default_rng(3)
    n, S, Q, B = 40, 200, 60, 96
    xy = torch.from_numpy(rng.uniform(0, 100, (n + 1, 2)).astype(np.float32)).cuda()
    tour = torch.from_numpy((rng.permutation(n) + 1).astype(np.int32)).cuda()
    q = torch.from_numpy(rng.integers(1, 20, (S, n)).astype(np.int32)).cuda()
    s = api.SaaSearch(tour, xy, q, Q, B, seed=8)
    s.autotune()
    t0, timed = s.state()
    assert torch.equal(t0, tour)
    s.run(1)
    _, first = s.state()
    assert torch.equal(timed, first) and len(set(first.tolist())) > B // 2
    arcs = s.count_arcs()
    s.autotune()
    assert torch.equal(s.state()[1], first) and s.count_arcs() == arcs
    s.close()
