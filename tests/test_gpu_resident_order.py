"""What the resident pivot kernel's CTAs publish to each other -- rows of B^-1,
moved slots of A, the tabu list, the records -- arrives whole: solves of one
problem repeat bit for bit, pivot by pivot."""
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


# one polling warp, three and five; the tie scan and the tabu list; the warm-start repair
@pytest.mark.parametrize("kind,m,n,opts", [("real", 200, 300, {}), ("real", 701, 1203, {}), ("real", 2000, 2600, {}),
                                           ("degenerate", 256, 512, dict(tol_tie=1e-6)), ("repair", 500, 700, {})])
def test_solves_repeat(kind, m, n, opts):
    from paper_1803_04378_gb300 import lpgb
    A, b, c = lpgen.degenerate_lp(m, n, 3) if kind == "degenerate" else lpgen.dense_real_lp(m, n, 3)
    with lpgb.LP(A, b, c, engine=2, trace_cap=1 << 14, max_iters=1500, **opts) as lp:
        first = None
        for _ in range(8):
            lp.reset()
            if kind == "repair":
                # every row's own column basic: many negative basic values to repair
                lp.set_basis_repair(np.arange(m, dtype=np.int32), 4 * m)
            res = lp.solve()
            assert res.persistent == 2
            t = lp.trace()
            now = (np.array([res.status, res.iterations]), t["q"], t["r"], t["theta"], t["dq"], t["flags"], *lp.state())
            if first is None:
                first = now
                if kind == "repair":
                    assert res.warm_repairs > 0
            assert all(np.array_equal(u, v) for u, v in zip(first, now))
