"""The warm-start network on batches of more than 65535 x 32 rows: more tiles of rows than
a grid's second dimension holds.

One input, one hidden unit and one output, with parameters and inputs that are small
powers of two: every product and activation is exact in FP16, so the logits are
exact.  The loss adds equal terms log 2 / B, but for one row of 0.03 / B: a tile's sum
passes through 17 FP32 additions after a logarithm of a few ulp, the tiles' sums are
added in FP64, so it is within 3e-6 of log 2.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

B = 65535 * 32 + 33


def test_more_rows_than_a_grid_dimension():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_04378_gb300 import lpgb
    net = lpgb.MLP(1, 1, 1, B)
    # W1 b1 W2 b2 W3 b3
    net.set_params(np.array([1.0, 0.0, 2.0, 0.5, 1.0, -1.0], np.float32))
    X = torch.full((B, 1), 0.25, device="cuda")
    X[-1] = 2.0
    T = torch.ones(B, 1, device="cuda")
    z = torch.empty(B, 1, device="cuda")
    net.forward(X, z)
    torch.cuda.synchronize()
    assert bool((z[:-1] == 0.0).all()) and float(z[-1]) == 3.5  # 2 x + 0.5 - 1
    _, loss = net.gradients(X, T)
    assert abs(loss - np.log(2.0)) <= 3e-6
    net.close()
