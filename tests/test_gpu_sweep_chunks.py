"""Sweeps whose planes a block leave remainders, against the oracle (needs a GB300)."""
import os

import numpy as np
import pytest

from oracle import multigrid as OM
from oracle.poisson import NEUMANN, PERIODIC

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


# (nx, ny, nz): 3D tiles of 32 x 8 and 64 x 8 and ragged ones, 2D rows of 256 and
# 128 and ragged ones; few planes, a prime number of them, many
SHAPES = [(96, 16, 31), (64, 8, 3), (192, 64, 67), (120, 72, 53), (40, 6, 7), (200, 24, 2), (256, 1, 5), (128, 1, 3),
          (384, 1, 53), (512, 1, 131), (360, 1, 37), (40, 1, 7), (300, 1, 997)]


@pytest.mark.parametrize("n", SHAPES)
@pytest.mark.parametrize("order", [0, 1])
def test_sweep_chunks(lm, n, order):
    """One float32 sweep, from zero and from a random x, against the oracle's float64
    sweep on the float32-rounded coefficients."""
    rng = np.random.default_rng(sum(n) + order)
    shape, h, bc = (n[2], n[1], n[0]), (1 / 64,) * 3, (PERIODIC, PERIODIC, NEUMANN)
    N = n[0] * n[1] * n[2]
    ct = (0.05 + rng.random(N)).astype(np.float32).astype(np.float64)
    rho = (0.5 + rng.random(N)).astype(np.float32).astype(np.float64)
    level = OM.build_hierarchy(ct.reshape(shape), rho.reshape(shape), h, bc)[0]
    f, x0 = rng.standard_normal(N).astype(np.float32), rng.standard_normal(N).astype(np.float32)
    d = lambda a: torch.as_tensor(a, device="cuda")
    with lm.Grid(n, h, bc) as g:
        g.set_coefficients_raw(ct, rho)
        out = torch.empty(N, dtype=torch.float32, device="cuda")
        for x in (None, x0):
            xin = np.zeros(N) if x is None else x.astype(np.float64)
            ref = OM.sweep(level, xin.reshape(shape), f.astype(np.float64).reshape(shape), "RB" if order == 0 else "BR")
            g.mg_sweep(None if x is None else d(x), d(f), out, order)
            got = out.cpu().numpy().astype(np.float64)
            assert np.linalg.norm(got - ref.ravel()) <= 1e-5 * np.linalg.norm(ref)
