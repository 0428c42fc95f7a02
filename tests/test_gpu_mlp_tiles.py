"""The batched network at the edges of its 128-row tiles, from aligned inputs
(full tiles arrive by bulk copies) and from inputs that start off 16 bytes
(plain loads): every output within the bound of test_gpu_mlp.py against the
FP64 network with the same BF16 roundings, and the two paths equal.  A
gradient over a partial last tile, and generated stencils against explicit
shapes, at the sizes where their loops end."""
import numpy as np
import pytest

from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("the GPU tests need a CUDA device")
    from paper_1908_04262_gb300 import build as B
    from paper_1908_04262_gb300 import lbf as L

    B.build()
    return L, torch


# 608 tiles fill the GPU once (four CTAs on each of 152 SMs): 77,824 rows
@pytest.mark.parametrize("n", [1, 127, 128, 129, 255, 256, 77824, 77825, 155777])
def test_forward_tiles(env, n):
    L, torch = env
    rng = np.random.default_rng(n)
    th = (mlp.init_params(4) + 0.05 * rng.normal(size=mlp.NPARAM)).astype(np.float32).astype(np.float64)
    x = rng.random((n, 27)).astype(np.float32)
    theta = torch.tensor(th, dtype=torch.float32, device="cuda")
    out = []
    for lead in (0, 1):  # rows are 108 bytes: the second start is off 16 bytes
        buf = torch.empty(n + lead, 27, device="cuda")
        xs = buf[lead:]
        xs.copy_(torch.tensor(x))
        y = torch.full((n + 1,), 7.0, device="cuda")
        L.mlp_forward(theta, xs, y[:n])
        torch.cuda.synchronize()
        assert y[n].item() == 7.0
        out.append(y[:n].cpu().numpy())
    assert np.array_equal(out[0], out[1])
    yb = mlp.forward_bf16(th, x.astype(np.float64))
    d = np.abs(out[0].astype(np.float64) - yb)
    W1, b1, W2, b2, W3, b3 = mlp.split(th)
    h2 = mlp.silu(mlp.silu(x @ W1.T + b1) @ W2.T + b2)
    assert np.mean(d <= 1e-5 * (1 + np.abs(yb))) >= 0.99
    assert np.all(d <= 2.0 ** -8 * (np.abs(h2) @ np.abs(W3)) + 1e-5)


@pytest.mark.parametrize("n", [1, 3, 4, 5, 33, 130])
def test_generated_fill_levels_match_sampling(env, n):
    """Fill levels are counts of sub-points: equal to the FP64 sampling of
    the same shapes, up to the order of the axes."""
    L, torch = env
    rng = np.random.default_rng(n)
    P = np.zeros((n, 20))
    want = []
    for i in range(n):
        R = np.exp(rng.uniform(np.log(2), np.log(40)))
        axes = R * (rng.uniform(0.75, 1.25, 3) if i % 2 else np.ones(3))
        q, r = np.linalg.qr(rng.normal(size=(3, 3)))
        q = q * np.sign(np.diag(r))
        c, d = rng.random(3), rng.normal(size=3)
        d /= np.linalg.norm(d)
        A = q @ np.diag(1 / axes ** 2) @ q.T
        cell = np.floor(c + d / np.sqrt(d @ A @ d) + 0.5)
        P[i, 0:3], P[i, 3:6], P[i, 6:15], P[i, 15], P[i, 16:19] = c, axes, q.ravel(), float(i % 3 > 0), cell
        want.append(np.sort(mlp.ellipsoid_stencil(c, axes, q, i % 3 > 0, cell)[0]))
    x, y = torch.empty(n, 27, device="cuda"), torch.empty(n, device="cuda")
    L.mlp_stencils_from_params(P, x, y)
    got = np.sort(x.cpu().numpy(), axis=1)
    assert np.array_equal(got, np.array(want).astype(np.float32))


def gradient_with_roundings(th, x, t):
    """Loss and gradient in FP64 with the operands of every product rounded
    to BF16 as the kernel rounds them."""
    r = mlp.bf16
    W1, b1, W2, b2, W3, b3 = mlp.split(th)
    n = len(x)
    X, V1, V2 = r(x), r(W1), r(W2)
    z1 = X @ V1.T + b1
    H1 = r(mlp.silu(z1))
    z2 = H1 @ V2.T + b2
    H2 = r(mlp.silu(z2))
    e = H2 @ W3 + b3[0] - t
    d3 = e / n
    d2 = r(d3[:, None] * W3 * mlp.dsilu(z2))
    d1 = r((d2 @ V2) * mlp.dsilu(z1))
    parts = [d1.T @ X, d1.sum(0), d2.T @ H1, d2.sum(0), H2.T @ d3, [d3.sum()]]
    return 0.5 * np.mean(e * e), np.concatenate([np.ravel(p) for p in parts])


@pytest.mark.parametrize("n", [1, 63, 65, 127, 128, 129, -5])
def test_gradient_tiles(env, n):
    """The gradient where the 128-row tiles end, and (n = -5) over two tiles
    and a partial third of every CTA.  What is left against the same BF16
    roundings in FP64 is FP32 sums (1e-5 of a block) and operands that round
    the other way, 2^-8 of one in a few hundred: 2e-3 of a block's norm."""
    L, torch = env
    if n < 0:
        n = 2 * 128 * torch.cuda.get_device_properties(0).multi_processor_count - n
    rng = np.random.default_rng(n)
    th = (mlp.init_params(6) + 0.05 * rng.normal(size=mlp.NPARAM)).astype(np.float32).astype(np.float64)
    x = rng.random((n, 27)).astype(np.float32).astype(np.float64)
    # residuals away from zero, more of one sign: no block cancels
    t = (mlp.forward(th, x) + rng.uniform(1, 2, n) * np.where(rng.random(n) < 0.8, 1, -1)).astype(np.float32).astype(np.float64)
    dev = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")  # noqa: E731
    grad = torch.full((mlp.NPARAM + 1,), 3.0, device="cuda")
    loss = torch.full((1,), 3.0, dtype=torch.float64, device="cuda")
    L.mlp_loss_grad(dev(th), dev(x), dev(t), grad[:-1], loss)
    g = grad.cpu().numpy().astype(np.float64)
    assert g[-1] == 3.0
    want_loss, want = gradient_with_roundings(th, x, t)
    assert abs(loss.item() - want_loss) < 2e-3 * want_loss
    k = 0
    for s in mlp.SIZES:
        m = int(np.prod(s))
        assert np.linalg.norm(g[k:k + m] - want[k:k + m]) < 2e-3 * np.linalg.norm(want[k:k + m]), s
        k += m
