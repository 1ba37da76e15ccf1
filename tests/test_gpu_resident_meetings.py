"""Steps of the resident pivot kernel that hold every meeting a step can hold.

Twenty copies of every column overflow the candidate lists, so that the FP64
pricing meets again, and a wide tie band lets the smallest ratios of several
CTAs tie, so that the tie set is scanned between two more.  A launch must not
reach meeting numbers that the next one begins with; at launches of one and
two pivots a number too many shows at once, at 64 only after a long run of such steps.

The bars are those of tests/test_gpu_resident.py: the dense engine's pivots and
flags, state within 1e-9 of its largest entry.
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


# (rows, columns before copying, tie band, rules): one polling warp, and three
@pytest.mark.parametrize("shape", [(60, 200, 0.3, {}), (150, 300, 1.0, dict(tabu_tenure=0, bland_after=0))])
@pytest.mark.parametrize("graph_iters", [1, 2, 64])
def test_every_meeting_in_a_step(shape, graph_iters):
    from paper_1803_04378_gb300 import lpgb
    m, n, band, rules = shape
    A, b, c = lpgen.dense_real_lp(m, n, 5)
    perm = np.random.default_rng(20).permutation(20 * n)
    A, c = np.tile(A, (1, 20))[:, perm], np.tile(c, 20)[perm]
    runs = []
    for engine in (0, 2):
        with lpgb.LP(A, b, c, engine=engine, trace_cap=1 << 10, max_iters=200, tol_tie=band, graph_iters=graph_iters,
                     **rules) as lp:
            res = lp.solve()
            runs.append((res, lp.trace(), *lp.solution(), lp.state()[1]))
    (r0, t0, x0, y0, z0, b0), (r1, t1, x1, y1, z1, b1) = runs
    assert r0.persistent == 1 and r1.persistent == 2
    assert r0.status == r1.status and r0.iterations == r1.iterations == 200
    assert np.array_equal(t0["q"], t1["q"]) and np.array_equal(t0["r"], t1["r"])
    assert np.array_equal(t0["flags"], t1["flags"])
    for u, v in ((x0, x1), (y0, y1), (b0, b1), (np.array([z0]), np.array([z1]))):
        assert np.max(np.abs(u - v)) <= 1e-9 * max(1.0, np.max(np.abs(u)))
