"""lp_price_static at duals that are zero on most rows (the list of nonzero duals)
and just past the limit of that list, against the reduced costs in FP64 by torch:
the same column (the draws leave no near ties), d_q to 1e-12 of the sum's size."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(1, 5), (3, 40), (4, 7), (33, 300), (515, 700), (4096, 333), (12288, 40)])
@pytest.mark.parametrize("extra", [None, 0, 1, "all"])
def test_sparse_duals(m, n, extra):
    """extra None: one nonzero dual; 0: as many as the list holds (m / 4); 1: one more."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_04378_gb300 import lpgb
    g = torch.Generator(device="cuda").manual_seed(m + n)
    lda = m + (m & 1) + 2
    A = torch.full((n, lda), float("nan"), dtype=torch.float64, device="cuda")
    A[:, :m] = torch.rand(n, m, generator=g, device="cuda", dtype=torch.float64)
    k = {None: 1, 0: m // 4, 1: min(m, m // 4 + 1), "all": m}[extra]
    y = torch.zeros(m, dtype=torch.float64, device="cuda")
    y[torch.randperm(m, generator=g, device="cuda")[:k]] = \
        torch.rand(k, generator=g, device="cuda", dtype=torch.float64) * (2.0 / max(1, k))
    c = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    pos = torch.full((n + m,), -1, dtype=torch.int32, device="cuda")
    pos[torch.randperm(n + m, generator=g, device="cuda")[:m]] = torch.arange(m, dtype=torch.int32, device="cuda")
    q = torch.full((1,), -7, dtype=torch.int32, device="cuda")
    dq = torch.zeros(1, dtype=torch.float64, device="cuda")
    rc = lpgb.price_static(m, n, A, lda, c, y, pos, 1e-9, q, dq, torch.cuda.current_stream().cuda_stream)
    assert rc == lpgb.LP_OK
    d = torch.cat([c - A[:, :m] @ y, -y])
    d[pos >= 0] = -np.inf
    best, j = d.max(0)
    assert abs(float(dq) - float(best)) <= 1e-12 * (1.0 + float(y.sum()))
    assert int(q) == (int(j) if float(best) > 1e-9 else -1)
