"""The cooperative Jacobi-PCG kernel at the edges of its cell-to-thread
mappings (warps dealt out, 2, 4 and 8 blocks of cells a block, one launch an
iteration past them), vs the oracle's PCG: iterates, history, iteration limit."""
import os

import numpy as np
import pytest

from oracle import poisson as P

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


# Float64 on both sides, the same recurrence: residuals of the first tens of
# iterations agree to rounding times the iteration count (1e-12), the solution
# to the tolerance of the solve times the condition of this diagonal-heavy
# system (below 10).
@pytest.mark.parametrize("n,bc", [
    ((1, 1, 1), (PER, PER, WALL)),
    ((3, 1, 11), (WALL, PER, WALL)),                 # one warp and a cell
    ((256, 1, 1), (PER, PER, WALL)),
    ((257, 1, 151), (PER, PER, WALL)),               # 38,807 cells: 152 blocks of cells
    ((255, 1, 152), (WALL, PER, WALL)),              # 38,760 cells: warps dealt out over the SMs
    ((51, 23, 67), (PER, PER, WALL)),                # four blocks of cells a block
    ((75, 45, 91), (PER, WALL, WALL)),               # 307,125 cells: eight
    ((75, 45, 93), (PER, PER, PER)),                 # 313,875 cells: past the kernel
])
def test_jacobi_pcg(lm, n, bc):
    rng = np.random.default_rng(n[0] + n[2])
    shape, h = (n[2], n[1], n[0]), (1 / 32, 1 / 24, 1 / 40)
    ct, rho = 400.0 + 4000.0 * rng.random(shape), 0.5 + rng.random(shape)
    f = rng.standard_normal(shape)
    op = P.Operator(ct, rho, h, bc)
    x, hist = np.zeros(shape), [1.0]
    dinv = 1.0 / op.diagonal()
    r, fn = f.copy(), np.linalg.norm(f)
    z = dinv * r
    p, rz = z.copy(), float((r * z).sum())
    while hist[-1] > 1e-10 and len(hist) < 400:
        q = op.apply(p)
        a = rz / float((p * q).sum())
        x += a * p
        r -= a * q
        hist.append(np.linalg.norm(r) / fn)
        z = dinv * r
        new = float((r * z).sum())
        p = z + new / rz * p
        rz = new
    g = lm.Grid(n, h, bc)
    g.set_coefficients_raw(ct.ravel(), rho.ravel())
    g.set_rhs(f.ravel())
    res = g.solve(mode="jacobi", rtol=1e-10)
    got, gh = g.solution(), g.residual_history()
    assert res["rel_residual"] <= 1e-10 and res["iters"] == len(hist) - 1 == len(gh) - 1
    np.testing.assert_allclose(gh[:20], hist[:20], rtol=1e-10, atol=1e-13)
    assert np.linalg.norm(got - x.ravel()) <= 1e-9 * np.linalg.norm(x)
    if len(hist) > 4:                                # the limit ends it after exactly that many iterations
        cut = g.solve(mode="jacobi", rtol=1e-10, max_iter=3, allow=(-3,))
        assert cut["status"] == -3 and cut["iters"] == 3
        again = g.solve(mode="jacobi", rtol=1e-10, check_every=1)
        assert again["iters"] == res["iters"] and np.array_equal(g.solution(), got)
    g.close()
