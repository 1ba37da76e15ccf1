"""lp_price_static around the list of the rows with a dual: the largest m (two blocks share
an SM's shared memory), the smallest m with a list, list lengths at the lines between the two passes (m / 4 where
warps have several columns, m / 8 where none has a second), runs of rows that end
inside a warp's 32, signed zeros and NaN among the duals.

Both passes add at most m products of at most one: 1e-12 (1 + sum |y|) bounds their
difference from torch's sum.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _price(m, n, k, seed, special=False):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_04378_gb300 import lpgb
    g = torch.Generator(device="cuda").manual_seed(seed)
    lda = m + (m & 1)
    A = torch.rand(n, lda, generator=g, device="cuda", dtype=torch.float64)
    y = torch.zeros(m, dtype=torch.float64, device="cuda")
    at = torch.randperm(m, generator=g, device="cuda")[:k]
    y[at] = torch.rand(k, generator=g, device="cuda", dtype=torch.float64) - 0.5
    if special:
        y[y == 0.0] = -0.0
    c = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    pos = torch.full((n + m,), -1, dtype=torch.int32, device="cuda")
    q = torch.full((1,), -7, dtype=torch.int32, device="cuda")
    dq = torch.zeros(1, dtype=torch.float64, device="cuda")
    rc = lpgb.price_static(m, n, A, lda, c, y, pos, 1e-9, q, dq, torch.cuda.current_stream().cuda_stream)
    assert rc == lpgb.LP_OK
    d = torch.cat([c - A[:, :m] @ y, -y])
    best, j = d.max(0)
    assert abs(float(dq) - float(best)) <= 1e-12 * (1.0 + float(y.abs().sum()))
    assert int(q) == (int(j) if float(best) > 1e-9 else -1)


@pytest.mark.parametrize("n", [3, 700, 9000])
@pytest.mark.parametrize("m", [12288, 12287, 10401, 513, 512, 511, 33, 7])
@pytest.mark.parametrize("part", [4, 8])
def test_both_sides_of_the_lines(m, n, part):
    for k in (m // part, min(m, m // part + 1)):
        _price(m, n, k, m + n + k)


def test_signed_zeros():
    _price(1000, 2000, 60, 5, special=True)


def test_nan_dual_is_not_passed_over():
    """A NaN among the duals makes every structural column's reduced cost NaN: no column improves."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_04378_gb300 import lpgb
    m, n = 100, 50
    A = torch.ones(n, m, dtype=torch.float64, device="cuda")
    y = torch.zeros(m, dtype=torch.float64, device="cuda")
    y[17] = float("nan")
    pos = torch.full((n + m,), -1, dtype=torch.int32, device="cuda")
    pos[n:] = torch.arange(m, dtype=torch.int32, device="cuda")
    q = torch.full((1,), -7, dtype=torch.int32, device="cuda")
    dq = torch.zeros(1, dtype=torch.float64, device="cuda")
    c = torch.ones(n, dtype=torch.float64, device="cuda")
    assert lpgb.price_static(m, n, A, m, c, y, pos, 1e-9, q, dq, torch.cuda.current_stream().cuda_stream) == lpgb.LP_OK
    assert int(q) == -1
