"""The cooperative Jacobi-PCG kernel against the iteration's own launches
(check_every = 1): the same bits whatever the iterations a launch, over restarts
and past the host's check; and a wait that runs out."""
import os
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PER, WALL = 0, 1


@pytest.fixture(scope="module")
def lm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1112_3507_gb300 import build as B
    if not os.path.exists(B.LIB) or any(os.path.getmtime(s) > os.path.getmtime(B.LIB) for s in B.sources()):
        B.build()
    from paper_1112_3507_gb300 import lowmach
    return lowmach


def _grid(lm, n, bc, ct, seed=0):
    rng = np.random.default_rng(seed)
    N = n[0] * n[1] * n[2]
    g = lm.Grid(n, (1 / 32, 1 / 24, 1 / 40), bc)
    g.set_coefficients_raw(ct * (1.0 + rng.random(N)), 0.5 + rng.random(N))
    g.set_rhs(rng.standard_normal(N))
    g.set_initial_guess(0.01 * rng.standard_normal(N))
    return g


def _solve(g, **kw):
    r = g.solve(mode="jacobi", allow=(0, -3), **kw)
    return r["status"], r["iters"], r["rel_residual"], g.solution(), g.residual_history()


def _same(a, b):
    assert a[:3] == b[:3] and np.array_equal(a[3], b[3]) and np.array_equal(a[4], b[4])


# Each mapping of cells to threads.  1e-10 ends by itself; the second tolerance
# lies below what the true residual reaches, so that the recurrence's
# convergence is followed by the restarts.
@pytest.mark.parametrize("n,bc", [
    ((129, 1, 97), (PER, PER, WALL)), ((255, 1, 152), (WALL, PER, WALL)), ((257, 1, 151), (PER, PER, WALL)),
    ((51, 23, 67), (PER, PER, WALL)), ((75, 45, 91), (PER, WALL, WALL)),
])
@pytest.mark.parametrize("rtol,use_x0", [(1e-10, 0), (2e-17, 1)])
def test_launches(lm, n, bc, rtol, use_x0):
    with _grid(lm, n, bc, 400.0) as g:
        kw = dict(rtol=rtol, use_x0=use_x0, max_iter=900)
        want = _solve(g, check_every=1, **kw)
        _same(_solve(g, **kw), want)
        for steps in (1, 7):
            g.jacobi_run_limits(steps=steps)
            _same(_solve(g, **kw), want)
        if rtol < 1e-16:                             # the recurrence passed it, the true residual did not
            assert want[0] == -3 and want[4].min() <= rtol < want[2]


def test_past_one_launch(lm):
    with _grid(lm, (2600, 1, 5), (WALL, PER, WALL), 1e-3) as g:
        g.solve(mode="jacobi", rtol=0.5)             # the inverse diagonal is formed once
        n0 = lm.kernel_launches()
        want = _solve(g, rtol=1e-11, check_every=1)
        n1 = lm.kernel_launches()
        _same(_solve(g, rtol=1e-11), want)
        n2 = lm.kernel_launches()
        assert want[0] == 0 and want[1] > 1100
        assert n1 - n0 > 3 * want[1] and n2 - n1 < 40


def test_a_wait_that_runs_out(lm):
    with _grid(lm, (129, 1, 97), (PER, PER, WALL), 400.0) as g:
        want = _solve(g, rtol=1e-10)
        g.jacobi_run_limits(looks=0)
        assert g.solve(mode="jacobi", rtol=1e-10, allow=(-5,))["status"] == -5
        g.jacobi_run_limits()
        _same(_solve(g, rtol=1e-10), want)


def test_solves_of_several_threads(lm):
    """Grids of their own on streams of their own: cooperative kernels beside each other."""
    sizes, bad = [(129, 1, 97), (257, 1, 151), (51, 23, 67), (64, 1, 64)], []

    def work(k):
        with torch.cuda.stream(torch.cuda.Stream()), _grid(lm, sizes[k], (PER, PER, WALL), 400.0, seed=k) as g:
            want = _solve(g, rtol=1e-10, check_every=1)
            for _ in range(20):
                got = _solve(g, rtol=1e-10)
                if got[:3] != want[:3] or not np.array_equal(got[3], want[3]):
                    bad.append(k)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
