"""Refinements past the sliced products' largest block, and with the slices off: the FP64
products with plain sums.

On these LPs the first k rows are live from the start and B11 = k I + E with 0 <= E <= 1:
its condition number is below 4 in the maximum norm, so products of length k and the
updates between two reinversions stay within 8 k 2^-52 of the elimination's inverse
(relative to its largest entry): below 4e-12 at k = 1500.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_04378_gb300 import lpgb  # noqa: F401


def _live(m, n, k):
    rng = np.random.default_rng(k)
    A = rng.random((m, n))
    A[np.arange(k), np.arange(k)] += k
    basis = np.arange(n, n + m, dtype=np.int32)
    basis[:k] = np.arange(k)
    x = np.zeros(n)
    x[:k] = 1.0 + rng.random(k)
    b = A @ x
    b[k:] += 1.0 + rng.random(m - k)
    return A, b, rng.random(n), basis


@pytest.mark.parametrize("m,k,tc", [(700, 300, 0), (1000, 511, 0), (1900, 1040, 1), (4096, 1500, 1)])
def test_plain_sums(m, k, tc):
    """The elimination's inverse, for a like number of operations."""
    from paper_1803_04378_gb300 import lpgb
    A, b, c, basis = _live(m, m + 100, k)
    runs = []
    for refine in (1, 0):
        with lpgb.LP(A, b, c, reinvert_refine=refine, reinvert_tc=tc, reinvert_every=16, max_iters=32,
                     trace_cap=64) as lp:
            lp.set_basis(basis)
            lp.solve()  # (kernels loaded)
            lp.set_basis(basis)
            res = lp.solve()
            runs.append((res, lp.trace(), *lp.state()))
    (r1, t1, B1, v1), (r0, t0, B0, v0) = runs
    assert r1.iterations == r0.iterations == 32 and r1.refined_reinversions == 2 and r0.refined_reinversions == 0
    assert np.array_equal(t1["q"], t0["q"]) and np.array_equal(t1["r"], t0["r"])
    assert np.max(np.abs(B1 - B0)) <= 8 * m * 2.0 ** -52 * np.max(np.abs(B0))
    assert np.max(np.abs(v1 - v0)) <= 8 * m * 2.0 ** -52 * np.max(np.abs(v0)) * np.max(np.abs(b)) / np.min(np.abs(b))
    # two of the three rebuilds are refinements there: 2 k^3 operations each, an elimination's
    # k^3 in smaller pieces (compensated sums, 5 k^3, took the three 1.96 times as long at k = 1500)
    assert r1.reinvert_gj_seconds < 1.5 * r0.reinvert_gj_seconds
