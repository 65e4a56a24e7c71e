"""The network's gradients against the float64 oracle where the arithmetic can
be followed exactly: small integer inputs and weights, so that every stored
activation is an exact BF16 integer on both sides."""
import os

import numpy as np
import pytest

from oracle import unet as U

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1112_3507_gb300 import build as B
    if not os.path.exists(B.LIB) or any(os.path.getmtime(s) > os.path.getmtime(B.LIB) for s in B.sources()):
        B.build()
    from paper_1112_3507_gb300 import lowmach
    return lowmach


def _bf16(a):
    return torch.as_tensor(np.asarray(a, dtype=np.float32)).to(torch.bfloat16).to(torch.float64).numpy()


# The output layer and D0 see the float32 gradient of the loss itself: their
# sums over n pixels in float32 chains of a few dozen steps stay within
# sqrt(n) 2^-24 / sqrt(n) times a small factor: 2e-6.  Every layer below adds
# one split-BF16 convolution (16 bits, 1.5e-5) to the gradient's error, at most
# eleven of them: 1.7e-4, times the cancellation of a bias or weight sum (< 4).
@pytest.mark.parametrize("ch,B,H,W", [
    ((16, 32, 48, 64), 2, 64, 48),       # every tensor-core width, whole tiles
    ((16, 32, 48, 64), 3, 40, 24),       # ragged tiles in both directions, an odd batch
    ((8, 16, 24, 32), 1, 8, 8),          # one-pixel coarsest level, half chunks of input channels
    ((4, 8, 12, 20), 2, 16, 56),         # four channels a thread, widths without a tensor-core chunk
    ((5, 8, 8, 16), 1, 24, 16),          # one channel a thread
    ((64, 64, 64, 64), 1, 16, 16),       # the widest chunks at every level
])
def test_gradients(lm, ch, B, H, W):
    rng = np.random.default_rng(B * H + W)
    P = U.init_params(rng, cin=3, ch=ch)
    for k, v in P.items():
        if v.ndim == 1:
            v[:] = 0.0
        elif k == "O":
            v[:] = rng.standard_normal(v.shape)
        else:
            v[:] = (rng.random(v.shape) < 2.5 / np.prod(v.shape[:-1])) * rng.choice([-1, 1, 1], v.shape)
    x = rng.integers(0, 4, (B, H, W, 3)).astype(np.float64)
    gy = rng.standard_normal((B, H, W, 1)).astype(np.float32)
    net = lm.Net(ch)
    net.set_params(U.flat_params(P, 3, ch))
    y = torch.empty(B * H * W, device="cuda")
    net.forward(torch.as_tensor(x.astype(np.float32).ravel(), device="cuda"), y, B, H, W)
    gyd = torch.as_tensor(gy.ravel(), device="cuda")
    net.backward(gyd)
    flat = net.grads()
    net.backward(gyd)
    assert np.array_equal(flat, net.grads())                     # fixed order of every sum
    net.close()
    Q = {k: (_bf16(v) if k[0] in "ABCD" else np.float32(v).astype(np.float64)) for k, v in P.items()}
    ref, cache = U.forward(Q, x, ch, rnd=_bf16)
    assert np.linalg.norm(y.cpu().numpy() - ref.ravel()) <= 1e-6 * max(np.linalg.norm(ref), 1.0)
    G, _ = U.backward(Q, cache, gy.astype(np.float64), ch)
    g = U.unflat_params(flat, 3, ch)
    for n, _ in U.param_shapes(3, ch):
        tol = 2e-6 if n in ("O", "o", "D0", "d0") else 7e-4
        assert np.linalg.norm(g[n] - G[n]) <= tol * np.linalg.norm(G[n]) + 1e-6, n


@pytest.mark.parametrize("n", [1, 1023, 1025, 70001])
def test_mse(lm, n):
    rng = np.random.default_rng(n)
    y, t = rng.standard_normal(n).astype(np.float32), rng.standard_normal(n).astype(np.float32)
    net = lm.Net((4, 8, 8, 8))
    yd, td = torch.as_tensor(y, device="cuda"), torch.as_tensor(t, device="cuda")
    gy = torch.empty_like(yd)
    for _ in range(2):                                           # the arrival counter is re-armed
        loss = net.mse(yd, td, gy)
        d = (y - t).astype(np.float64)
        assert abs(loss - np.mean(d * d)) <= 1e-12 * np.mean(d * d) + 1e-300
        np.testing.assert_allclose(gy.cpu().numpy(), 2.0 * d / n, rtol=2e-7, atol=0)
    net.close()
