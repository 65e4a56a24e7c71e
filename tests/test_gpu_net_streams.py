"""The network's calls on streams of their own: losses beside a busy default
stream and from several threads, and passes captured in graphs."""
import os
import threading

import numpy as np
import pytest

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


def _pair(n, seed):
    rng = np.random.default_rng(seed)
    y, t = rng.standard_normal(n).astype(np.float32), rng.standard_normal(n).astype(np.float32)
    d = (y - t).astype(np.float64)
    return torch.as_tensor(y, device="cuda"), torch.as_tensor(t, device="cuda"), float(np.mean(d * d))


def test_first_loss_beside_a_busy_default_stream(lm):
    """What the loss's reduction starts from is in place whatever the default stream has queued."""
    y, t, want = _pair(200001, 1)
    gy, s = torch.empty_like(y), torch.cuda.Stream()
    torch.cuda.synchronize()
    net = lm.Net((4, 8, 8, 8))
    torch.cuda._sleep(50_000_000)                    # some 25 ms on the default stream
    for _ in range(3):
        assert abs(net.mse(y, t, gy, stream=s) - want) <= 1e-12 * want
    torch.cuda.synchronize()
    assert abs(net.mse(y, t, gy, stream=s) - want) <= 1e-12 * want
    net.close()


def test_losses_of_one_net_from_several_threads(lm):
    net, bad = lm.Net((4, 8, 8, 8)), []

    def work(k):
        with torch.cuda.stream(torch.cuda.Stream()):
            y, t, want = _pair(100001 + 4096 * k, k)
            gy = torch.empty_like(y)
            torch.cuda.current_stream().synchronize()
            for _ in range(50):
                got = net.mse(y, t, gy)
                if not abs(got - want) <= 1e-12 * want:
                    bad.append((k, got, want))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    net.close()
    assert not bad


def _net(lm, seed, ch=(16, 32, 48, 64)):
    net = lm.Net(ch)
    p = np.random.default_rng(seed).standard_normal(net.nparams).astype(np.float32) * 0.1
    net.set_params(p)
    return net, p


@pytest.mark.parametrize("ch", [(16, 32, 48, 64), (5, 8, 12, 16)])
def test_captured_passes_follow_the_weights(lm, ch):
    """A captured forward and backward pass, replayed after the weights changed, gives what eager passes give."""
    B, H, W = 2, 32, 24
    net, p = _net(lm, 3, ch)
    x = torch.randn(B * H * W * 3, device="cuda")
    gy = torch.randn(B * H * W, device="cuda")
    y, ye = torch.empty(B * H * W, device="cuda"), torch.empty(B * H * W, device="cuda")

    def passes(out):
        net.forward(x, out, B, H, W)
        net.backward(gy)

    side = torch.cuda.Stream()
    with torch.cuda.stream(side):                    # buffers are allocated by the first passes
        passes(y)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        passes(y)
    for change in (lambda: net.adam(0.05), lambda: net.set_params(-p)):
        change()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        got = net.grads()
        passes(ye)
        torch.cuda.synchronize()
        assert torch.equal(y, ye) and np.array_equal(got, net.grads())
    del graph
    net.close()


def test_a_capture_leaves_eager_passes_their_weights(lm):
    """A pass captured right after the weights changed has run nothing: eager passes still see the new weights."""
    B, H, W = 1, 32, 32
    net, p = _net(lm, 4)
    x = torch.randn(B * H * W * 3, device="cuda")
    y, ye, yw = (torch.empty(B * H * W, device="cuda") for _ in range(3))
    net.forward(x, y, B, H, W)
    net.set_params(2.0 * p)
    net.forward(x, yw, B, H, W)                      # what the new weights give
    net.set_params(p)
    net.forward(x, ye, B, H, W)
    torch.cuda.synchronize()
    net.set_params(2.0 * p)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        net.forward(x, y, B, H, W)
    net.forward(x, ye, B, H, W)
    torch.cuda.synchronize()
    assert torch.equal(ye, yw)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, yw)
    del graph
    net.close()
