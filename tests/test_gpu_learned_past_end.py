"""The parameter gradient where a tile's rows past the end would have infinite activations or products
of their own (needs a GB300): a hidden unit that every row switches off and zero inputs switch on,
with an infinite output weight, or with a finite path whose value overflows.  All other parameters,
inputs and gradients are small integers, so the gradient is exact, as in 64 bits over the rows that
there are.  The row counts reach several tiles per block and chunks of the greatest length."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _gradient(X, theta, d):
    W1, b1, W2, b2, W3, b3 = np.split(theta.astype(np.float64), np.cumsum([1024, 64, 4096, 64, 128]))
    W1, W2, W3 = W1.reshape(64, 16), W2.reshape(64, 64), W3.reshape(2, 64)
    h1 = np.maximum(X @ W1.T + b1, 0)
    h2 = np.maximum(h1 @ W2.T + b2, 0)
    on = h2 > 0
    assert not on[:, 0].any()                            # the unit with the infinite weight
    d2 = np.where(on, d @ np.where(np.isfinite(W3), W3, 0), 0)
    d1 = (d2 @ W2) * (h1 > 0)
    parts = [(d1, X), (d1, None), (d2, h1), (d2, None), (d, h2), (d, None)]
    size = max(float((np.abs(a).T @ np.abs(b) if b is not None else np.abs(a).sum(0)).max()) for a, b in parts)
    return np.concatenate([(a.T @ b if b is not None else a.sum(0)).ravel() for a, b in parts]), size


@pytest.mark.parametrize("huge", ["weight", "overflow"])
@pytest.mark.parametrize("n", [1, 63, 65, 19457, 83073, 311297])
def test_rows_past_the_end_add_nothing(n, huge):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2608_30239_gb300 import learned, mcpd
    ctx = mcpd.Context(0)
    rng = np.random.default_rng(n)
    sparse = lambda k, p: rng.integers(-1, 2, k) * (rng.random(k) < p)        # noqa: E731
    W1, W2, W3 = sparse(1024, 0.5).astype(np.float32), sparse(4096, 0.1).astype(np.float32), sparse(128, 0.5).astype(np.float32)
    b1, b2, b3 = (sparse(k, 0.5).astype(np.float32) for k in (64, 64, 2))
    top = 1.0 if huge == "weight" else 2.0 ** 127
    W1[:16], b1[0] = 0, top                              # unit 0 of the first layer: top - top x_0
    W1[0] = -top
    W2[:64], b2[0] = 0, 0                                # unit 0 of the second: twice that
    W2[0] = 2.0
    W3[0], W3[64] = (np.inf, 0.0) if huge == "weight" else (1.0, 1.0)
    theta = np.concatenate([W1, b1, W2, b2, W3, b3])
    X = rng.integers(-2, 3, (n, 16)).astype(np.float64)
    X[:, 0] = 1.0
    d = rng.integers(-1, 2, (n, 2)).astype(np.float64)
    d[rng.random(n) > 3000 / n] = 0.0
    d[-1] = 1.0
    grad, size = _gradient(X, theta, d)
    assert size < 2 ** 24
    W = torch.from_numpy(theta).cuda().bfloat16()
    Xd, dd = (torch.from_numpy(a.astype(np.float32)).cuda() for a in (X, d))
    L, p = learned._lib(), learned._p
    need = int(L.mcpd_mlp_backward_workspace(n))
    work = torch.full((need,), float("nan"), device="cuda:0")
    got = torch.full((theta.size,), float("nan"), device="cuda:0")
    torch.cuda.synchronize()
    assert L.mcpd_mlp_backward(ctx.h, n, p(Xd), p(W), p(dd), p(work), need, p(got)) == 0
    torch.cuda.synchronize()
    assert np.array_equal(got.cpu().numpy(), grad)
    ctx.close()
