"""The one-launch coarse V-cycle (levels in one block, shared by the blocks of
a cluster, with and without a dense inverse at the bottom) vs the oracle's
float64 V-cycle on the float32-rounded coefficients."""
import os

import numpy as np
import pytest

from oracle import multigrid as OM

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


# One float32 cycle against the float64 one: each half-sweep rounds its values
# once (6e-8), a smoothing step does not amplify them and the exact or smoothed
# bottom returns them damped, so a few tens of half-sweeps stay below 1e-5; the
# bar is the V-cycle's 1e-4 of the parity tests.
@pytest.mark.parametrize("n,bc,nu", [
    ((64, 1, 64), (PER, PER, WALL), (2, 3)),         # 2048 pairs: the most one block takes
    ((64, 1, 66), (PER, PER, WALL), (2, 3)),         # just over: shared rows, an unsolved level of 64 x 33 rows
    ((200, 1, 130), (WALL, PER, WALL), (1, 2)),      # uneven shares of rows, odd coarse rows, unsolved bottom
    ((256, 1, 128), (PER, PER, PER), (2, 3)),        # two shared levels of 128-cell segments, wrapped in z
    ((45, 1, 25), (WALL, PER, WALL), (2, 3)),        # one unsolved level of odd rows
    ((1, 1, 40), (PER, PER, WALL), (3, 1)),          # rows of one cell
    ((2, 1, 6), (PER, PER, PER), (8, 8)),            # two-cell rows: both faces to one neighbour
    ((30, 18, 11), (PER, PER, WALL), (2, 3)),        # an unsolved level shared plane by plane
    ((24, 20, 28), (PER, PER, WALL), (2, 2)),        # 3D, shared, planes in twos
    ((24, 8, 30), (WALL, WALL, PER), (1, 1)),        # walls in x and y, wrapped in z
    ((20, 4, 2), (PER, PER, WALL), (2, 3)),          # few planes
])
def test_vcycle(lm, n, bc, nu):
    rng = np.random.default_rng(sum(n) * 7 + nu[0])
    shape, h = (n[2], n[1], n[0]), (1 / 64, 1 / 48, 1 / 80)
    ct = (0.05 + rng.random(shape)).astype(np.float32).astype(np.float64) * 50.0
    rho = (0.5 + rng.random(shape)).astype(np.float32).astype(np.float64)
    r = rng.standard_normal(shape).astype(np.float32)
    levels = OM.build_hierarchy(ct, rho, h, bc, coarse_max=16)
    ref = OM.vcycle(levels, r.astype(np.float64), nu1=nu[0], nu2=nu[1], coarse_max=64).ravel()
    g = lm.Grid(n, h, bc)
    g.set_coefficients_raw(ct.ravel(), rho.ravel())
    rd = torch.as_tensor(r.ravel(), device="cuda")
    z, again = torch.empty_like(rd), torch.full_like(rd, 7.0)
    before = lm.kernel_launches()
    g.mg_vcycle(rd, z, *nu)
    g.mg_vcycle(rd, again, *nu)
    assert torch.equal(z, again)
    assert [tuple(reversed(L.shape)) for L in levels] == g.mg_levels()
    assert lm.kernel_launches() - before <= 2 + len(levels) + 2      # coarsening, inverse and plan, then a launch a cycle
    # new coefficients through the same handle: the plan follows them
    g.set_coefficients_raw(ct.ravel() * 3.0, rho.ravel())
    g.mg_vcycle(rd, again, *nu)
    g.close()
    assert not torch.equal(z, again)
    z = z.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(z - ref) <= 1e-4 * np.linalg.norm(ref)
