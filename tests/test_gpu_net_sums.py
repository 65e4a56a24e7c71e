"""The network's float64 sums at the ends of float32's range: losses and bias
gradients whose terms or partial sums no float32 holds, and infinities."""
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


# A sum of n positive terms in float64: a thread's few dozen, a tree of eight
# steps in a block and one over the blocks stay below 64 roundings of 2^-53.
@pytest.mark.parametrize("n", [7, 300007])
@pytest.mark.parametrize("scale", [1e-30, 1e-22, 1.0, 1e25, 1e38])
def test_loss(lm, n, scale):
    rng = np.random.default_rng(n)
    y, t = ((0.5 + rng.random(n)) * s * scale for s in (1.0, -1.0))
    y, t = y.astype(np.float32), t.astype(np.float32)
    d = (y - t).astype(np.float64)
    net = lm.Net((4, 8, 8, 8))
    yd, td = torch.as_tensor(y, device="cuda"), torch.as_tensor(t, device="cuda")
    want = np.mean(d * d)
    assert abs(net.mse(yd, td, torch.empty_like(yd)) - want) <= 64 * 2.0 ** -53 * want
    net.close()


def _net(lm, ch):
    """D0 passes its channels through, C0 the sum of the upsampled and the skip ones; the other convolutions give their bias, 1."""
    P = U.init_params(np.random.default_rng(0), cin=3, ch=ch)
    for k, v in P.items():
        v[:] = 1.0 if v.ndim == 1 or k == "O" else 0.0
    for c in range(ch[0]):
        P["D0"][1, 1, c, c] = P["C0"][1, 1, c, c] = P["C0"][1, 1, ch[1] + c, c] = 1.0
    net = lm.Net(ch)
    net.set_params(U.flat_params(P, 3, ch))
    return net


def _grads(lm, ch, n, gy):
    net = _net(lm, ch)
    net.forward(torch.zeros(3 * n * n, device="cuda"), torch.empty(n * n, device="cuda"), 1, n, n)
    net.backward(torch.as_tensor(gy, device="cuda"))
    g = U.unflat_params(net.grads(), 3, ch)
    net.close()
    return g


# Gradients of 2^e, the first half of the pixels positive, the second negative
# and the last zero: the sum is 2^e, and a thread's share of either half is
# past float32's range.  (Where 2^125 is, d1's four fine pixels add up to 2^127;
# 2^127 there would not be a float32, nor what the encoder below gets from it.)
@pytest.mark.parametrize("names,n,e", [(("o", "d0", "c0"), 1024, 127), (("o", "d0", "c0", "b0", "d1"), 2048, 125)])
def test_bias_gradients_past_float32(lm, names, n, e):
    gy = np.full(n * n, 2.0 ** e, dtype=np.float32)
    gy[n * n // 2:] *= -1
    gy[-1] = 0.0
    g = _grads(lm, (8, 8, 8, 8), n, gy)
    for k in names:
        assert np.all(g[k] == 2.0 ** e), k


def test_infinite_gradient(lm):
    gy = np.ones(512 * 512, dtype=np.float32)
    gy[100 * 512 + 77] = np.inf                      # inside: no zero beside it
    g = _grads(lm, (8, 8, 8, 8), 512, gy)
    for k in ("o", "O", "d0", "D0"):
        assert np.all(g[k] == np.inf), k


# One cut of a tile's sum (below 2^-23 of it, always to one side), and random
# roundings of 2^-24 in some two dozen additions a warp and group: 2^-23 + 5 2^-24.
@pytest.mark.parametrize("B,n", [(1, 64), (16, 256)])
def test_weight_gradient_of_one_sign(lm, B, n):
    ch = (8, 8, 8, 8)
    P = U.init_params(np.random.default_rng(0), cin=3, ch=ch)
    for k, v in P.items():
        v[:] = 1.0 if k in ("O", "d0") else 0.0
    for c in range(8):                               # D0's input is the image's channel c % 3
        P["A0"][1, 1, c % 3, c] = P["B0"][1, 1, c, c] = P["C0"][1, 1, 8 + c, c] = 1.0
    g = torch.Generator(device="cuda").manual_seed(B)
    x = torch.rand((B, n, n, 3), device="cuda", generator=g).mul_(0.9).add_(0.1).to(torch.bfloat16).float()
    gy = torch.rand((B, n, n), device="cuda", generator=g).add_(0.5)
    net = lm.Net(ch)
    net.set_params(U.flat_params(P, 3, ch))
    net.forward(x.reshape(-1), torch.empty(gy.numel(), device="cuda"), B, n, n)
    net.backward(gy.reshape(-1))
    got = U.unflat_params(net.grads(), 3, ch)["D0"]
    net.close()
    xp = torch.nn.functional.pad(x.double(), (0, 0, 1, 1, 1, 1))
    for t in range(9):
        want = (xp[:, t // 3:t // 3 + n, t % 3:t % 3 + n] * gy.double()[..., None]).sum((0, 1, 2)).cpu().numpy()
        want = want[np.arange(8) % 3][:, None]
        assert np.all(np.abs(got[t // 3, t % 3] - want) <= 7 * 2.0 ** -24 * want), t
