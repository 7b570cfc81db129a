"""The FP64 mean of costs whose spread exceeds what a pair of floats holds.
One thread's group of eight is the same for all 256 threads of the one block,
so the tree and the division by 2,048 are exact and at most the group's seven
FP64 additions round: 7 x 2^-53 of the sum (all values are positive), 8 with
the rounding of the reference."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GROUPS = [
    [705625054, 9718, 18, 6293060, 2519793, 456674, 96, 25],            # 2^25
    [16, 371302060, 11, 15685, 8240455, 1684, 6, 36],                   # 2^26
    [1 << 30, 1, 3, 5, 7, 11, 13, 17],                                  # 2^30
    [1 << 19, 1, 3, 5, 7, 11, 13, 17],                                  # 19 exponents: the pair's last
    [1 << 20, 1, 3, 5, 7, 11, 13, 17],                                  # 20: the first beyond it
    [437758252, 0, 0, 28532968, 0, 26386848, 0, 1],                     # zeros do not count
    [0, 0, 0, 0, 0, 0, 0, 3],
]


@pytest.mark.parametrize("group", range(len(GROUPS)))
@pytest.mark.parametrize("p", [0.1, 1.0e-20, 3.0e-39])  # the last: costs below the least normal float
def test_mean_over_a_wide_spread(group, p):
    from paper_2602_05179_gb300 import api
    d = np.repeat(np.asarray(GROUPS[group], np.int32)[:, None], 256, 1).reshape(-1, 1)
    zero = torch.zeros(1, device="cuda")
    r = api.reinsert_eval(1, 0, 0, 0.0, p, 0.0, zero, torch.from_numpy(d).cuda())
    v = r["value"].cpu().numpy().astype(np.float64)
    assert v.shape == (2048,) and (v[d[:, 0] > 0] > 0).any()
    exact = math.fsum(v) / 2048
    assert abs(float(r["mean"]) - exact) <= 8 * 2.0 ** -53 * exact
