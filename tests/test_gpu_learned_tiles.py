"""The tiled MLP kernels at row counts around their tiles (64 rows) and chunks (whole tiles, one up
to ceil(n / 304) rows), needs a GB300.  Parameters, inputs and gradients are small integers, so
every product and sum is exact in fp32 (below 2^24 in magnitude, checked) and in any order: the
kernels must give the 64-bit values exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _reference(X, theta, d):
    W1, b1, W2, b2, W3, b3 = np.split(theta.astype(np.float64), np.cumsum([1024, 64, 4096, 64, 128]))
    W1, W2, W3 = W1.reshape(64, 16), W2.reshape(64, 64), W3.reshape(2, 64)
    h1 = np.maximum(X @ W1.T + b1, 0)
    h2 = np.maximum(h1 @ W2.T + b2, 0)
    d2 = (d @ W3) * (h2 > 0)
    d1 = (d2 @ W2) * (h1 > 0)
    parts = [(d1, X), (d1, None), (d2, h1), (d2, None), (d, h2), (d, None)]
    grad = np.concatenate([(a.T @ b if b is not None else a.sum(0)).ravel() for a, b in parts])
    size = max(float((np.abs(a).T @ np.abs(b) if b is not None else np.abs(a).sum(0)).max()) for a, b in parts)
    return h2 @ W3.T + b3, grad, size


@pytest.mark.parametrize("n", [1, 63, 64, 65, 1298, 19457])
def test_row_counts_around_tiles_and_chunks(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2608_30239_gb300 import learned, mcpd
    ctx = mcpd.Context(0)
    rng = np.random.default_rng(n)
    sparse = lambda k, p: rng.integers(-1, 2, k) * (rng.random(k) < p)        # noqa: E731
    theta = np.concatenate([sparse(1024, 0.5), sparse(64, 0.5), sparse(4096, 0.1), sparse(64, 0.5), sparse(128, 0.5),
                            sparse(2, 0.5)]).astype(np.float32)
    X = rng.integers(-2, 3, (n, 16)).astype(np.float64)
    d = rng.integers(-1, 2, (n, 2)).astype(np.float64)
    out, grad, size = _reference(X, theta, d)
    assert size < 2 ** 24 and np.abs(out).max() < 2 ** 24
    model = learned.MLP(ctx, seed=0)
    model.master.copy_(torch.from_numpy(theta))
    model.cast()
    Xd, dd = (torch.from_numpy(a.astype(np.float32)).cuda() for a in (X, d))
    assert np.array_equal(model.forward(Xd).cpu().numpy(), out)
    need = int(learned._lib().mcpd_mlp_backward_workspace(n))
    work = torch.full((need,), float("nan"), device="cuda:0")
    model.grad.fill_(float("nan"))
    rc = learned._lib().mcpd_mlp_backward(ctx.h, n, learned._p(Xd), learned._p(model.W), learned._p(dd),
                                          learned._p(work), need, learned._p(model.grad))
    assert rc == 0
    assert np.array_equal(model.grad.cpu().numpy(), grad)
    ctx.close()


@pytest.mark.parametrize("x_off,w_off", [(0, 1), (1, 0), (3, 5)])
def test_arrays_off_their_16_byte_boundary(x_off, w_off):
    """The C ABI takes any float rows and bf16 parameters: off the boundary of the wide loads too."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2608_30239_gb300 import learned, mcpd
    ctx = mcpd.Context(0)
    n, rng = 131, np.random.default_rng(7)
    theta = (rng.integers(-1, 2, 5378) * (rng.random(5378) < 0.2)).astype(np.float32)
    X = rng.integers(-2, 3, (n, 16)).astype(np.float64)
    d = rng.integers(-1, 2, (n, 2)).astype(np.float64)
    out, grad, size = _reference(X, theta, d)
    assert size < 2 ** 24 and np.abs(out).max() < 2 ** 24
    xs = torch.zeros(n * 16 + x_off, device="cuda:0")
    ws = torch.zeros(theta.size + w_off, dtype=torch.bfloat16, device="cuda:0")
    xs[x_off:] = torch.from_numpy(X.astype(np.float32).ravel()).cuda()
    ws[w_off:] = torch.from_numpy(theta).cuda().bfloat16()
    L, p = learned._lib(), learned._p
    dd, got = torch.from_numpy(d.astype(np.float32)).cuda(), torch.empty((n, 2), device="cuda:0")
    need = int(L.mcpd_mlp_backward_workspace(n))
    work, g = torch.empty(need, device="cuda:0"), torch.empty(theta.size, device="cuda:0")
    torch.cuda.synchronize()
    assert L.mcpd_mlp_forward(ctx.h, n, p(xs[x_off:]), p(ws[w_off:]), p(got)) == 0
    assert L.mcpd_mlp_backward(ctx.h, n, p(xs[x_off:]), p(ws[w_off:]), p(dd), p(work), need, p(g)) == 0
    torch.cuda.synchronize()
    assert np.array_equal(got.cpu().numpy(), out) and np.array_equal(g.cpu().numpy(), grad)
    ctx.close()
