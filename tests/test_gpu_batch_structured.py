"""The batch kernel's slack-structured pivots where their paths part: screened
columns that tie (more than the selection's list holds), every number of re-priced
candidates, slots that join, leave and move, reinversions within a few pivots, each
block size.  Bars as in tests/test_gpu_batch.py: every pivot valid to the oracle
(follow mode; relaxed under the BF16 screen), objectives and certificates to 1e-9."""
import numpy as np
import pytest

import lpgen
import oracle
from gpu_util import assert_certificate

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


def _problems():
    rng = np.random.default_rng(4)
    probs = []
    A, b, c = lpgen.dense_real_lp(40, 9, 5)
    for copies in (4, 50):  # 36 and 450 columns, each LP's screen full of exact ties
        perm = rng.permutation(9 * copies)
        probs.append((np.ascontiguousarray(np.tile(A, (1, copies))[:, perm]), b, np.tile(c, copies)[perm]))
    probs.append(lpgen.degenerate_lp(33, 65, 3))   # slacks re-enter: slots leave and move
    probs.append(lpgen.degenerate_lp(127, 129, 4))
    probs.append(lpgen.dense_int_lp(5, 3, 1))      # fewer columns than candidates
    probs.append(lpgen.dense_real_lp(256, 512, 2))
    probs.append(lpgen.dense_real_lp(129, 31, 2))
    return probs


@pytest.mark.parametrize("opts", [dict(), dict(topk=1), dict(topk=3), dict(reinvert_every=3), dict(price_mode=0),
                                  dict(bland_after=2), dict(tabu_tenure=200)])
@pytest.mark.parametrize("threads", [128, 256, 512])
def test_pivots_valid(opts, threads):
    from paper_1803_04378_gb300 import lpgb
    probs = _problems()
    with lpgb.Batch(probs, trace_cap=4096, max_iters=3000, **opts) as bt:
        bt.set_tuning([threads, 1, threads, 0, threads, 0, threads, 0])
        bt.solve()
        st, it, obj, xs, ys = bt.results()
        for k, (A, b, c) in enumerate(probs):
            tr = bt.trace(k)
            o = oracle.Options(**{v: opts[v] for v in ("reinvert_every", "bland_after", "tabu_tenure") if v in opts},
                               follow_relaxed=0 if opts.get("price_mode") == 0 else 1, max_iters=3000)
            q, r = tr["q"], tr["r"]
            if st[k] == 1:
                q, r = np.append(q, -1), np.append(r, -1)
            chk = oracle.solve(A, b, c, o, follow=(q, r))
            assert chk.mismatch_at < 0 and chk.iterations == it[k], (k, chk.mismatch_at)
            if st[k] == 1:
                ref = oracle.solve(A, b, c)
                assert abs(obj[k] - ref.objective) <= 1e-9 * max(1.0, abs(ref.objective)), k
                assert_certificate(A, b, c, xs[k], ys[k])
        assert np.count_nonzero(st == 1) >= 5
