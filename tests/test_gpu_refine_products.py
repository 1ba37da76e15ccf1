"""The refinement's products in FP64 and in 7-bit slices, at the edges of their tiles, of
the chunks of 64 columns and of the rule between them (needs a GB300).

On these LPs every pivot brings in a structural variable for its own row's slack, so the
reinversion at pivot k refines a k x k block.  B11 = 10 I + E with 0 <= E <= 5 / m has a
condition number below 3 in the maximum norm, so the rounding of two products of length
k <= 171 and of up to 171 updates stays below 3 * 2 * 171 * 2^-52 * 4 < 1e-12.
"""
import numpy as np
import pytest

from gpu_util import gpu_solve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("engine", [0, 2])
@pytest.mark.parametrize("k", [1, 7, 8, 63, 64, 65, 128, 171])
def test_refined_inverse_matches_elimination(engine, k):
    m = 300
    rng = np.random.default_rng(k)
    A = 10.0 * np.eye(m) + rng.random((m, m)) * (5.0 / m)
    b, c = 1.0 + rng.random(m), 1.0 + rng.random(m)
    states = []
    for refine, tc in ((1, 1), (1, 0), (0, 0)):
        lp, res, *_ = gpu_solve(A, b, c, engine=engine, reinvert_every=k, reinvert_refine=refine, reinvert_tc=tc,
                                max_iters=k)
        assert res.iterations == k and res.reinversions == 1 and res.refined_reinversions == refine
        assert np.sum(lp.basis() < m) == k
        states.append(lp.state())
        lp.close()
    for binv, bbar in states[:2]:
        assert np.max(np.abs(binv - states[2][0])) <= 1e-12
        assert np.max(np.abs(bbar - states[2][1])) <= 1e-12 * np.max(np.abs(b))
