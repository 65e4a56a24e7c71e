"""The convolutions' variants at images large enough for the launches to choose
them: every width of output channels, one and two pixel rows a warp, weight
gradients of several tiles a group with a short last group and ragged tiles."""
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


def _round(v):
    """BF16 storage, gradients passed through."""
    return v + (v.detach().to(torch.bfloat16).double() - v.detach())


def _reference(P, x, gy, ch):
    """(y, gradients) of the network in float64 with its stored activations in BF16."""
    F = torch.nn.functional
    p = {k: torch.as_tensor(np.asarray(v, dtype=np.float64), device="cuda").requires_grad_() for k, v in P.items()}

    def conv(v, k):
        return _round(F.relu(F.conv2d(v, p[k].permute(3, 2, 0, 1), p[k.lower()], padding=1)))

    v, skips = x.double().permute(0, 3, 1, 2), []
    for l in range(4):
        v = v if l == 0 else _round(F.avg_pool2d(v, 2))
        v = conv(conv(v, f"A{l}"), f"B{l}")
        skips.append(v)
    for l in (2, 1, 0):
        v = conv(conv(torch.cat((F.interpolate(v, scale_factor=2, mode="nearest"), skips[l]), 1), f"C{l}"), f"D{l}")
    y = torch.einsum("bchw,co->bhw", v, p["O"]) + p["o"]
    y.backward(gy.double())
    return y.detach(), {k: t.grad.cpu().numpy() for k, t in p.items()}


# Blocks at level 0 are 16 x 8 pixels, 418 of them in 2 x 152 x 168 (more than
# two an SM: the widest chunk of the channels) and 1386 in 3 x 264 x 216 (eight
# an SM: two rows a warp up to 32 channels); coarser levels take narrower ones.
# Weight gradients: 3 to 14 tiles a group, the last group short.  Small integer
# inputs and sparse weights of +-1, so stored activations are the same on both
# sides; below D0 a gradient has passed up to eleven split-BF16 convolutions of
# 16 bits each, times the cancellation of a sum (< 4).
@pytest.mark.parametrize("ch,B,H,W", [
    ((64, 8, 8, 8), 2, 152, 168), ((56, 8, 8, 8), 2, 152, 168), ((48, 16, 8, 8), 2, 152, 168),
    ((40, 8, 8, 8), 2, 152, 168), ((32, 8, 8, 8), 2, 152, 168), ((16, 8, 8, 8), 2, 152, 168),
    ((32, 16, 8, 8), 3, 264, 216), ((16, 32, 48, 64), 3, 264, 216), ((8, 8, 16, 16), 3, 264, 216),
])
def test_gradients(lm, ch, B, H, W):
    rng = np.random.default_rng(ch[0] + H)
    P = U.init_params(rng, cin=3, ch=ch)
    for k, v in P.items():
        if v.ndim == 1:
            v[:] = 0.0
        elif k == "O":
            v[:] = np.float32(rng.standard_normal(v.shape))
        else:
            v[:] = (rng.random(v.shape) < 2.5 / np.prod(v.shape[:-1])) * rng.choice([-1, 1, 1], v.shape)
    x = torch.as_tensor(rng.integers(0, 4, (B, H, W, 3)).astype(np.float32), device="cuda")
    gy = torch.as_tensor(rng.standard_normal((B, H, W)).astype(np.float32), device="cuda")
    net = lm.Net(ch)
    net.set_params(U.flat_params(P, 3, ch))
    y = torch.empty(gy.numel(), device="cuda")
    net.forward(x.reshape(-1), y, B, H, W)
    net.backward(gy.reshape(-1))
    got = U.unflat_params(net.grads(), 3, ch)
    net.close()
    ref, G = _reference(P, x, gy, ch)
    assert float((y - ref.reshape(-1)).norm()) <= 1e-6 * max(float(ref.norm()), 1.0)
    for n, _ in U.param_shapes(3, ch):
        tol = 2e-6 if n in ("O", "o", "D0", "d0") else 7e-4
        assert np.linalg.norm(got[n] - G[n]) <= tol * np.linalg.norm(G[n]) + 1e-6, n
