"""sdp_reinsert_workspace_bytes does not depend on value0_out: a caller may size
its workspace once and ask for C_0(I) in some of the calls."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu  # the lane kernel's part is a number of bytes per SM


def _args(api, T, U, K=0, algo=0, S=64, policy=4096, value0=None):
    a = api.ReinsertArgs()
    a.T, a.U, a.I0, a.algo, a.S, a.n_routes = T, U, U // 2, algo, S, K
    a.h, a.p, a.unit_cost = 1.0, 2.0, 0.0
    a.policy_out, a.value0_out = policy, value0
    return a


@pytest.mark.parametrize("T,U,K", [(30, 100, 0), (30, 100, 4), (60, 200, 0), (60, 200, 8), (129, 200, 0),
                                   (30, 300, 0), (30, 1000, 0)])
@pytest.mark.parametrize("algo", [0, 1, 2])
def test_size_covers_both(T, U, K, algo):
    from paper_2602_05179_gb300 import api
    lib = api._load()
    for policy in (None, 4096):
        without, with_v0 = (_args(api, T, U, K, algo, policy=policy, value0=v) for v in (None, 4096))
        size = lib.sdp_reinsert_workspace_bytes(ctypes.byref(without))
        assert size == lib.sdp_reinsert_workspace_bytes(ctypes.byref(with_v0))
        for a in (without, with_v0):
            assert 4096 <= lib.sdp_reinsert_call_bytes(ctypes.byref(a)) <= size


def test_value0_in_a_workspace_sized_without_it():
    from paper_2602_05179_gb300 import api
    lib = api._load()
    T, U, S = 30, 100, 64
    cons = torch.randint(0, 9, (S, T), dtype=torch.int32, device="cuda")
    fixed = torch.full((T,), 5.0, device="cuda")
    ref = api.reinsert_eval(T, U, U // 2, 1.0, 2.0, 0.0, fixed, cons, value0=True, algo="warp")
    a = _args(api, T, U)
    val = torch.empty(S, device="cuda")
    pol = torch.empty((S, T), dtype=torch.uint8, device="cuda")
    v0 = torch.empty((S, U + 1), device="cuda")
    a.fixed, a.consumption = fixed.data_ptr(), cons.data_ptr()
    a.value_out, a.policy_out = val.data_ptr(), pol.data_ptr()
    ws = torch.empty(lib.sdp_reinsert_workspace_bytes(ctypes.byref(a)), dtype=torch.uint8, device="cuda")
    a.workspace, a.workspace_bytes = ws.data_ptr(), ws.numel()
    a.value0_out = v0.data_ptr()
    assert lib.sdp_reinsert_eval(ctypes.byref(a), None) == 0, lib.sdp_last_error()
    torch.cuda.synchronize()
    assert torch.equal(val, ref["value"]) and torch.equal(pol, ref["policy"]) and torch.equal(v0, ref["value0"])
