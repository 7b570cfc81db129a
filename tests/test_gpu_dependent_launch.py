"""The kernels of a call are placed while their predecessors run
(dependent.cuh): calls of different sizes back to back on one stream, alone
and replayed from a captured graph, return what each returns by itself."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _calls():
    from paper_2602_05179_gb300 import api
    rng = np.random.default_rng(8)
    cuda = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    out = []
    for n, S in ((50, 1000), (1, 1), (33, 32), (200, 4097), (50, 1000), (333, 6000)):
        tour = cuda((rng.permutation(n) + 1).astype(np.int32))
        q = cuda(rng.integers(0, 30, (S, n)).astype(np.int32))
        dist = cuda(rng.uniform(1, 9, (n + 1, n + 1)).astype(np.float32))
        for preds in ("u16", None):
            out.append(lambda t=tour, d=q, c=dist, p=preds: api.split_eval(t, 90, d, dist=c, preds=p))
        one = torch.ones((), device="cuda")
        out.append(lambda t=tour, d=q, c=dist, o=one: dict(grad=api.split_backward(t, 90, d, c, o)[0]))
    cons, fixed = cuda(rng.integers(0, 9, (1500, 30)).astype(np.int32)), cuda(rng.uniform(1, 9, 30).astype(np.float32))
    out.append(lambda: api.reinsert_eval(30, 100, 50, 1.0, 20.0, 0.5, fixed, cons))
    return out


def _same(a, b):
    return all(torch.equal(a[k].view(torch.uint8) if a[k].dim() else a[k], b[k].view(torch.uint8) if b[k].dim() else b[k])
               for k in a if a[k] is not None)


def test_back_to_back_equals_alone():
    calls = _calls()
    alone = []
    for f in calls:
        alone.append(f())
        torch.cuda.synchronize()
    for _ in range(4):
        got = [f() for f in calls]
        torch.cuda.synchronize()
        assert all(_same(a, g) for a, g in zip(alone, got))


def test_captured_equals_alone():
    calls = _calls()
    alone = [f() for f in calls]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = [f() for f in calls]
    for _ in range(3):
        for g in got:
            for v in g.values():
                if v is not None:
                    v.fill_(7)
        graph.replay()
        torch.cuda.synchronize()
        assert all(_same(a, g) for a, g in zip(alone, got))
