"""k_iterate_r against k_iterate_s, bit for bit.

A priority list takes the structured engine to k_iterate_s.  With every variable
listed its rule is Dantzig's over the non-tabu columns again, so the two kernels
have the same pivots to make; the order of every sum is the same too, and
with it the step lengths, reduced costs, B^-1, basic values, duals and objective.
Equality of numbers: -0 and 0 are one value.
"""
import numpy as np
import pytest

import lpgen

pytestmark = pytest.mark.gpu

TF_GUIDED = 128  # the priority list chose the entering variable


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_04378_gb300 import lpgb  # noqa: F401


def _live(m, n, k):
    """k of m rows live from the start."""
    rng = np.random.default_rng(4)
    A = rng.random((m, n)) + np.pad(np.eye(k) * k, ((0, m - k), (0, n - k)))
    basis = np.arange(n, n + m, dtype=np.int32)
    basis[:k] = np.arange(k)
    x = np.zeros(n)
    x[:k] = 1.0 + rng.random(k)
    b = A @ x
    b[k:] += 1.0 + rng.random(m - k)
    return A, b, rng.random(n), basis


# one CTA's rows and several CTAs'; A and B^-1 on chip, A alone, neither
SHAPES = [("int", 40, 60), ("real", 90, 150), ("real", 300, 421), ("real", 701, 1203), ("live", 1800, 2000, 1000),
          ("real", 100, 70000)]


@pytest.mark.parametrize("shape", SHAPES)
def test_bits_of_both_kernels(shape):
    from paper_1803_04378_gb300 import lpgb
    kind, m, n = shape[:3]
    basis = None
    if kind == "live":
        A, b, c, basis = _live(*shape[1:])
    else:
        A, b, c = lpgen.dense_int_lp(m, n, 3) if kind == "int" else lpgen.dense_real_lp(m, n, 3)
    runs = []
    for listed in (True, False):
        with lpgb.LP(A, b, c, engine=2, trace_cap=1 << 12, max_iters=300) as lp:
            if listed:
                lp.set_priority(np.arange(n + m, dtype=np.int32))
            if basis is not None:
                lp.set_basis(basis)
            res = lp.solve()
            assert res.persistent == 2
            x, y, z = lp.solution()
            runs.append((res.status, res.iterations, lp.trace(), x, y, z, *lp.state(), lp.basis()))
    s, r = runs
    assert s[:2] == r[:2] and r[1] > 0
    for key in ("q", "r", "theta", "dq"):
        assert np.array_equal(s[2][key], r[2][key]), key
    assert np.array_equal(s[2]["flags"] & ~TF_GUIDED, r[2]["flags"])
    for u, v in zip(s[3:], r[3:]):
        assert np.array_equal(np.asarray(u), np.asarray(v))
