"""Reinversion by refinement where most of the basis is structural (needs a GB300).

The refinement keeps three k x k blocks: in scratch of m^2 elements where 3 k^2 <= m^2, and in
scratch of its own up to k = 256.  On these LPs every pivot brings in a structural variable
for its own row's slack, so k runs from 0 to m: the periodic reinversions within either rule
are refined, the others eliminated, with the pivots of a run that eliminates throughout.

The bound on x and y: B11 = 10 I + E with |E| <= 5 / m has a condition number below 3 in
the maximum norm, and the sums have at most m terms: 3 m 2^-52 relative to the largest
entry, times 8 for the two runs' updates between reinversions, is below 1e-11 at m = 700.
"""
import numpy as np
import pytest

from gpu_util import assert_certificate, gpu_solve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,every", [(7, 2), (96, 16), (131, 8), (320, 32), (700, 50)])
def test_refined_up_to_all_structural(m, every):
    rng = np.random.default_rng(m)
    A = 10.0 * np.eye(m) + rng.random((m, m)) * (5.0 / m)
    b, c = 1.0 + rng.random(m), 1.0 + rng.random(m)
    lp1, r1, x1, y1, z1, t1 = gpu_solve(A, b, c, reinvert_every=every)
    lp0, r0, x0, y0, z0, t0 = gpu_solve(A, b, c, reinvert_every=every, reinvert_refine=0)
    assert r1.status == r0.status == 1 and r1.iterations == r0.iterations == m
    assert np.all(lp1.basis() < m)
    assert r0.refined_reinversions == 0 and r1.reinversions == r0.reinversions >= (m - 1) // every
    assert r1.refined_reinversions == sum(k <= 256 or 3 * k * k <= m * m
                                          for k in range(every, every * r1.reinversions + 1, every))
    assert np.array_equal(t1["q"], t0["q"]) and np.array_equal(t1["r"], t0["r"])
    assert np.max(np.abs(x1 - x0)) <= 1e-11 * np.max(np.abs(x0))
    assert np.max(np.abs(y1 - y0)) <= 1e-11 * np.max(np.abs(y0))
    assert_certificate(A, b, c, x1, y1)
    lp1.close()
    lp0.close()
