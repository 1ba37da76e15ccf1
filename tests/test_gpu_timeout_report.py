"""A wait that only one CTA gives up is reported, whichever CTA that is: the
self-test keeps a record from the last CTA, while the lead CTA gets all of its own."""
import time

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_04378_gb300 import lpgb  # noqa: F401


@pytest.mark.parametrize("blocks", [1, 2, 64])
def test_timeout_of_one_cta_is_reported(blocks):
    from paper_1803_04378_gb300 import lpgb
    t0 = time.time()
    assert lpgb.selftest_barrier_timeout(blocks) == lpgb.LP_ERR_TIMEOUT
    assert time.time() - t0 < 60
