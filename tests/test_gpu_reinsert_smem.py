"""Shapes whose rows fill a CTA's shared memory to within the kernel's own few
bytes: AUTO against the warp kernel, with as many warps as fit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,U", [(31, 721), (31, 736), (50, 500), (72, 400), (84, 300), (101, 250), (127, 100)])
def test_rows_that_fill_the_shared_memory(T, U):
    from paper_2602_05179_gb300 import api
    # the last U of the shape that still fits, a few below it and one above
    def need(u):
        return (((T + u + 1) * 4 + 15) // 16 * 16, (T + 1) * 32 * 14)
    S = 16 * 32 * torch.cuda.get_device_properties(0).multi_processor_count + 1
    rng = np.random.default_rng(T)
    cons = torch.from_numpy(rng.poisson(U / 5.0, (S, T)).astype(np.int32)).cuda()
    fixed = torch.from_numpy(rng.uniform(5, 50, T).astype(np.float32)).cuda()
    warps = (227 * 1024) // need(U)[1]
    edge = (227 * 1024 - need(U)[1] * warps) // 4 - T - 1  # the largest table beside that many warps
    for u in sorted({min(max(edge + k, 1), 1023) for k in (-17, -13, -9, -5, -4, -3, -1, 0, 1)} | {U}):
        table = torch.from_numpy(rng.uniform(0, 30, u + 1).astype(np.float32)).cuda()
        args = (T, u, u // 2, 1.25, 20.0, 0.0, fixed, cons)
        try:
            ref = api.reinsert_eval(*args, table=table, algo="warp")
        except api.SdpError as e:  # decision bits that no kernel holds (T x words above 4,096)
            assert e.code == -5
            continue
        r = api.reinsert_eval(*args, table=table)
        for key in ("value", "policy", "mean"):
            assert torch.equal(r[key], ref[key]), (u, key)
