"""The network's calls on streams of their own: losses beside a busy default
stream and from several threads."""
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
