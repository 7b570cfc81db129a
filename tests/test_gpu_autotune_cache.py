"""The autotuner's cache file: an entry serves the plans whose shapes stand for
the kernels it was timed with, and no others."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

B, N, S, Q = 64, 24, 64, 60


def _plan(shared):
    from paper_2602_05179_gb300 import api
    rng = np.random.default_rng(5)
    tours = np.stack([rng.permutation(N) + 1 for _ in range(B)]).astype(np.int32)
    xy = rng.uniform(0, 100, (N + 1, 2)).astype(np.float32)
    q = rng.integers(1, 20, (S, N)).astype(np.int32)
    dem = q if shared else np.tile(q, (B, 1))
    dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda()
           for x in (tours.reshape(-1), np.tile(xy, (B, 1)), dem.reshape(-1))]
    return api.SplitPlan([N] * B, *dev, Q, S, dem_off=[0] * B if shared else None)


def _lines(path):
    return path.read_text().splitlines()


def test_plans_on_one_and_on_many_demand_arrays_have_their_own_entries(tmp_path):
    path = tmp_path / "cache.txt"
    plans = [_plan(True), _plan(False)]
    shapes = [p.autotune(str(path)) for p in plans]
    keys = [line.split()[0] for line in _lines(path)]
    assert len(keys) == 2 and keys[0] != keys[1]
    for p, shape in zip(plans, shapes):  # both are hits now
        assert p.autotune(str(path)) == shape
        p.close()
    assert len(_lines(path)) == 2


def test_entries_without_the_kernels_do_not_match(tmp_path):
    path = tmp_path / "cache.txt"
    prop = torch.cuda.get_device_properties(0)
    key = (f"{prop.name}|sm{prop.multi_processor_count}|B{B}|S{S}|Q{Q}|nmax{N}|sumn{B * N}").replace(" ", "_")
    path.write_text(f"{key} 1 8 1\n")
    p = _plan(True)
    p.autotune(str(path))
    assert len(_lines(path)) == 2  # timed anew
    p.close()
