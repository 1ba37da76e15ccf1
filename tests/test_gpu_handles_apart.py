"""Handles of different sizes beside each other: what one is given must not
take from another what its launches need (a kernel's shared-memory limit
belongs to the kernel, not to the handle)."""
import threading

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


# engine, priority list, options, what must run (lp_result.persistent)
CASES = [(2, False, {}, 2), (2, True, {}, 2), (0, False, {}, 1), (1, False, {}, 0), (1, False, dict(price_mode=1), 0)]


@pytest.mark.parametrize("engine,prio,opts,kernel", CASES)
def test_small_handle_after_large(engine, prio, opts, kernel):
    """4200 rows: the vectors a block keeps are past the 48 KB that every kernel may use, in every engine."""
    from paper_1803_04378_gb300 import lpgb
    big, small = lpgen.dense_real_lp(4200, 300, 7), lpgen.dense_real_lp(40, 60, 7)
    with lpgb.LP(*big, engine=2, max_iters=20) as lp:
        want = lp.solve()
    with lpgb.LP(*big, engine=engine, max_iters=20, **opts) as lp, lpgb.LP(*small, engine=engine, **opts) as other:
        for h, A in ((lp, big[0]), (other, small[0])):
            if prio:
                h.set_priority(np.arange(sum(A.shape), dtype=np.int32))
        other.solve()
        got = lp.solve()
    assert got.persistent == kernel and got.engine_reason == 0
    assert got.iterations == want.iterations == 20
    if not opts:  # (price_mode 1 re-prices the top columns of a BF16 screen: other pivots may win ties)
        assert abs(got.objective - want.objective) <= 1e-9 * abs(want.objective)


def test_threads_of_two_sizes():
    """Two host threads, each with its own handle, solving over and over."""
    from paper_1803_04378_gb300 import lpgb
    out = {}

    def work(name, data):
        with lpgb.LP(*data) as lp:
            rs = []
            for _ in range(40):
                lp.reset()
                rs.append(lp.solve())
        out[name] = [(r.persistent, r.engine_reason, r.status, r.iterations, r.objective) for r in rs]

    jobs = [(k, lpgen.dense_real_lp(m, n, 11)) for k, m, n in (("a", 256, 512), ("b", 700, 1200))]
    ths = [threading.Thread(target=work, args=j) for j in jobs]
    for t in ths:
        t.start()
    for t in ths:
        t.join()
    for name, _ in jobs:
        assert len(set(out[name])) == 1, name  # every solve like the first
        assert out[name][0][:3] == (2, 0, 1)
