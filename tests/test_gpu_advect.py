"""The advection passes at the edges of their warps and chunks (needs a GB300)."""
import os

import numpy as np
import pytest

from oracle import fractional as FR
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


# (nz, ny, nx): rows around the 29 results of a warp, axes of one and two cells,
# columns around a thread's chunk (16 cells and 4)
SHAPES = [(2, 1, 2), (3, 2, 2), (40, 1, 1), (1, 1, 33), (5, 1, 26), (4, 3, 29), (7, 2, 31), (130, 1, 3), (17, 16, 58),
          (33, 5, 87), (96, 84, 88)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("bc", [(PERIODIC,) * 3, (NEUMANN,) * 3])
@pytest.mark.parametrize("with_c", [False, True])
def test_advect_edges(lm, shape, bc, with_c):
    rng = np.random.default_rng(sum(shape))
    n, h, dt = (shape[2], shape[1], shape[0]), (0.1, 0.2, 0.15), 0.01
    rho = 1.0 + 0.5 * rng.random(shape)
    mom = [rng.standard_normal(shape) for _ in range(3)]
    mom[1][...] = 0.0                                     # at rest along y
    mom[2][rng.random(shape) < 0.3] = 0.0
    e = 4.0 + 1e-9 * rng.random(shape)                    # nearly flat
    rc = rng.random(shape) * 2.0 ** rng.integers(-600, 1, shape) if with_c else None   # slopes whose product underflows
    ref_rho, ref_m, ref_e, ref_c = FR.advect(rho, mom, e, dt, h, bc, rho_c=rc)
    N = rho.size
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a).ravel(), dtype=torch.float64, device="cuda")
    r1, m1, e1 = d(np.zeros(N)), d(np.zeros(3 * N)), d(np.zeros(N))
    c1 = d(np.zeros(N)) if with_c else None
    lm.advect(n, h, bc, dt, d(rho), d(np.concatenate([m.ravel() for m in mom])), d(e), r1, m1, e1,
              rho_c=d(rc) if with_c else None, rho_c_new=c1)
    m1 = m1.cpu().numpy().reshape(3, *shape)
    pairs = [(ref_rho, r1.cpu().numpy(), rho), (ref_e, e1.cpu().numpy(), e)]
    pairs += [(ref_m[a], m1[a], mom[a]) for a in range(3)]
    if with_c:
        pairs.append((ref_c, c1.cpu().numpy(), rc))
    for ref, got, q0 in pairs:                            # rounding scale: dt / h times the flux magnitudes
        scale = np.abs(q0).max() * (1 + dt * 20.0 / min(h))
        np.testing.assert_allclose(got.reshape(shape), ref, rtol=0, atol=1e-14 * scale)
