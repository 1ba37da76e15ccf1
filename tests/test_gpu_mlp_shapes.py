"""The warm-start network at shapes where its tiles end raggedly -- widths off the
64-column K blocks, batches below a tile, past one and off its 8-row atoms, a
smaller batch after a larger one in the same handle -- bit for bit.

The data make every sum exact in FP32 whatever its order: features and weights are
small integers, six nonzeros per row or column.  For the gradients b3 cancels the
logits (the features that W1 uses are the same in every sample, the others are
not), so sigmoid is 1/2, dz3 is +-h with h the FP16 value of 1 / (2 B), dz2 and dz1
are integer multiples k h with k <= 36, and the weight gradients sums of at most 256
products below 2^24 h."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _sparse(rng, rows, cols, axis):
    """Integers in {-1, 1}, six per row (axis 1) or per column (axis 0), zero elsewhere."""
    W = np.zeros((rows, cols))
    n, m = (rows, cols) if axis == 1 else (cols, rows)
    for i in range(n):
        at = rng.choice(m, min(6, m), replace=False)
        W[(i, at) if axis == 1 else (at, i)] = rng.choice([-1.0, 1.0], len(at))
    return W


@pytest.mark.parametrize("dims,batches", [((6, 8, 5), [1, 3]), ((70, 40, 130), [33, 7, 64, 1]),
                                          ((320, 96, 129), [129, 256, 100]), ((1025, 513, 700), [256, 128, 9]),
                                          ((6144, 512, 3072), [256, 1])])
def test_exact(dims, batches):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1803_04378_gb300 import lpgb
    n_in, hid, out = dims
    rng = np.random.default_rng(sum(dims))
    W1, W2, W3 = _sparse(rng, n_in, hid, 0), _sparse(rng, hid, hid, 1), _sparse(rng, hid, out, 1)
    W1[n_in // 2:] = 0.0  # features that only the gradient of W1 sees
    b1, b2 = rng.integers(0, 3, hid).astype(float), rng.integers(0, 3, hid).astype(float)
    net = lpgb.MLP(n_in, hid, out, max(batches), torch.cuda.current_stream().cuda_stream)
    relu = lambda v: np.maximum(v, 0.0)  # noqa: E731
    half = lambda v: np.asarray(v, np.float64).astype(np.float16).astype(np.float64)  # noqa: E731
    for B in batches:
        # logits, every sample its own
        b3 = rng.integers(-2, 3, out).astype(float)
        net.set_params(np.concatenate([v.ravel() for v in (W1, b1, W2, b2, W3, b3)]))
        X = rng.integers(-2, 3, (B, n_in)).astype(float)
        z = relu(relu(X @ W1 + b1) @ W2 + b2) @ W3 + b3
        logits = torch.full((B, out), float("nan"), device="cuda")
        net.forward(torch.from_numpy(X).float().cuda(), logits)
        assert np.array_equal(logits.cpu().numpy(), z.astype(np.float32)), B
        # gradients at logits of zero
        X[:, :n_in // 2] = X[0, :n_in // 2]
        z1 = X @ W1 + b1
        a1 = relu(z1)
        z2 = a1 @ W2 + b2
        a2 = relu(z2)
        b3 = -(a2[0] @ W3)
        net.set_params(np.concatenate([v.ravel() for v in (W1, b1, W2, b2, W3, b3)]))
        T = (rng.random((B, out)) < 0.4).astype(float)
        d3 = half((0.5 - T).astype(np.float32) * (np.float32(1.0) / np.float32(B)))
        d2 = half(np.where(z2 > 0, d3 @ W3.T, 0.0))
        d1 = half(np.where(z1 > 0, d2 @ W2.T, 0.0))
        want = np.concatenate([v.ravel() for v in (X.T @ d1, d1.sum(0), a1.T @ d2, d2.sum(0), a2.T @ d3, d3.sum(0))])
        got, loss = net.gradients(torch.from_numpy(X).float().cuda(), torch.from_numpy(T).float().cuda())
        assert np.array_equal(got, want.astype(np.float32)), B
        assert abs(loss - out * np.log(2.0)) <= 1e-5 * out
    net.close()
