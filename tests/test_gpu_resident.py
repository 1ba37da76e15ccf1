"""The resident pivot kernel (k_iterate_r) where its paths part: several columns
whose FP32 intervals overlap, more of them than a record lists, ratio ties that
several CTAs share, no improving column the screen can prove, layouts that do not
hold A or B^-1 in shared memory, and live slots that outgrow a launch's layout.

The arithmetic is that of the dense engine up to the order of nonzero terms, so
the bars are those of tests/test_gpu_structured.py: the same pivots and flags,
state within 1e-9 of its largest entry.
"""
import numpy as np
import pytest

import lpgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_04378_gb300 import lpgb  # noqa: F401


def _same_as_dense(A, b, c, basis=None, **opts):
    from paper_1803_04378_gb300 import lpgb
    runs = []
    for engine in (0, 2):
        with lpgb.LP(A, b, c, engine=engine, trace_cap=1 << 14, **opts) as lp:
            if basis is not None:
                lp.set_basis(basis)
            res = lp.solve()
            runs.append((res, lp.trace(), *lp.solution(), lp.state()[1]))
    (r0, t0, x0, y0, z0, b0), (r1, t1, x1, y1, z1, b1) = runs
    assert r0.persistent == 1 and r1.persistent == 2
    assert r0.status == r1.status and r0.iterations == r1.iterations
    assert np.array_equal(t0["q"], t1["q"]) and np.array_equal(t0["r"], t1["r"])
    assert np.array_equal(t0["flags"], t1["flags"])
    for u, v in ((x0, x1), (y0, y1), (b0, b1), (np.array([z0]), np.array([z1]))):
        assert np.max(np.abs(u - v)) <= 1e-9 * max(1.0, np.max(np.abs(u)))
    return r1


@pytest.mark.parametrize("copies", [2, 3, 5, 40])
def test_equal_columns(copies):
    """Every column `copies` times: exact ties of d_j, resolved to the smallest
    index; 40 copies overflow the lists of the records and of the CTAs."""
    A, b, c = lpgen.dense_real_lp(90, 24, 5)
    perm = np.random.default_rng(copies).permutation(24 * copies)
    A, c = np.tile(A, (1, copies))[:, perm], np.tile(c, copies)[perm]
    _same_as_dense(A, b, c)


def test_ratio_ties_across_ctas():
    """Ratios that differ by less than tol_tie and lie in different CTAs (the rows
    are dealt to CTAs round-robin): the tie set is scanned over all rows."""
    A, b, c = lpgen.dense_int_lp(48, 60, 9)
    A[:, 0] = 1.0
    c[0] = 500.0
    b[:] = 1000.0 * (1.0 + 1e-13 * np.arange(48))
    r = _same_as_dense(A, b, c)
    assert r.tabu_pushes > 0


@pytest.mark.parametrize("opts", [dict(tabu_tenure=500), dict(tabu_tenure=0, bland_after=1), dict(bland_after=3),
                                  dict(reinvert_every=5), dict(tol_tie=1e-6)])
def test_rules(opts):
    """A tabu list that covers every improving column (aspiration), the safety net
    from the first degenerate pivots on, short reinversion periods, a wide tie band."""
    A, b, c = lpgen.degenerate_lp(70, 120, 3)
    _same_as_dense(A, b, c, max_iters=400, **opts)


def test_columns_past_shared_memory():
    """60000 columns: neither A nor B^-1 is held in shared memory."""
    A, b, c = lpgen.dense_real_lp(120, 60000, 6)
    _same_as_dense(A, b, c, max_iters=150)


def test_many_live_slots():
    """A start with 1000 of 1800 rows live: B^-1 does not fit in shared memory, and
    with a launch of 64 pivots the live slots pass a multiple of 64."""
    rng = np.random.default_rng(8)
    m, n, k = 1800, 2000, 1000
    A = rng.random((m, n)) + np.pad(np.eye(k) * k, ((0, m - k), (0, n - k)))
    basis = np.arange(n, n + m, dtype=np.int32)
    basis[:k] = np.arange(k)
    x = np.zeros(n)
    x[:k] = 1.0 + rng.random(k)
    b = A @ x
    b[k:] += 1.0 + rng.random(m - k)
    _same_as_dense(A, b, rng.random(n), basis=basis, max_iters=100)
