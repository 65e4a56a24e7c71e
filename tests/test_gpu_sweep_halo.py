"""Red-black sweeps and V-cycles of 3D grids whose tiles end in y beside an x
wall, or whose rows are single cells: the halo cells there take the first colour
like any other (vs the oracle's sweep and V-cycle)."""
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


def _problem(n, seed):
    rng = np.random.default_rng(seed)
    shape, h = (n[2], n[1], n[0]), (1 / 64, 1 / 48, 1 / 80)
    ct = (0.05 + rng.random(shape)).astype(np.float32).astype(np.float64) * 50.0
    rho = (0.5 + rng.random(shape)).astype(np.float32).astype(np.float64)
    return shape, h, ct, rho, rng.standard_normal(shape).astype(np.float32), rng.standard_normal(shape).astype(np.float32)


SIZES = [((10, 8, 33), (WALL, PER, WALL)), ((40, 24, 30), (WALL, PER, WALL)), ((71, 17, 20), (WALL, WALL, PER)),
         ((66, 20, 10), (WALL, PER, PER)), ((130, 40, 24), (WALL, WALL, WALL)), ((1, 16, 20), (PER, PER, WALL)),
         ((1, 30, 12), (WALL, WALL, WALL)), ((2, 24, 7), (PER, PER, WALL)), ((24, 20, 28), (PER, WALL, WALL)),
         ((64, 24, 20), (WALL, PER, WALL)), ((32, 16, 9), (WALL, WALL, WALL)), ((128, 32, 12), (WALL, PER, WALL)),
         ((256, 16, 9), (WALL, PER, WALL))]            # (whole tiles and rows: kernels of their own)


# One sweep in float32: each value is rounded a few times and seen by a
# neighbour once more, so 1e-6 of the norm; a V-cycle of some tens of half-sweeps
# the bar of the parity tests, 1e-4.
@pytest.mark.parametrize("n,bc", SIZES)
@pytest.mark.parametrize("first", [0, 1])
def test_sweep(lm, n, bc, first):
    shape, h, ct, rho, x, f = _problem(n, sum(n))
    with lm.Grid(n, h, bc) as g:
        g.set_coefficients_raw(ct.ravel(), rho.ravel())
        xd, fd = (torch.as_tensor(a.ravel(), device="cuda") for a in (x, f))
        out = torch.empty_like(xd)
        g.mg_sweep(xd, fd, out, first)
        got = out.cpu().numpy().astype(np.float64)
    ref = OM.sweep(OM.Level(ct, rho, h, bc), x.astype(np.float64), f.astype(np.float64), "RB" if first == 0 else "BR")
    assert np.linalg.norm(got - ref.ravel()) <= 1e-6 * np.linalg.norm(ref)


@pytest.mark.parametrize("n,bc", SIZES)
@pytest.mark.parametrize("nu", [(1, 1), (2, 3)])
def test_vcycle(lm, n, bc, nu):
    shape, h, ct, rho, r, _ = _problem(n, sum(n) + 1)
    levels = OM.build_hierarchy(ct, rho, h, bc, coarse_max=16)
    ref = OM.vcycle(levels, r.astype(np.float64), nu1=nu[0], nu2=nu[1], coarse_max=64).ravel()
    with lm.Grid(n, h, bc) as g:
        g.set_coefficients_raw(ct.ravel(), rho.ravel())
        rd = torch.as_tensor(r.ravel(), device="cuda")
        z = torch.empty_like(rd)
        g.mg_vcycle(rd, z, *nu)
        got = z.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - ref) <= 1e-4 * np.linalg.norm(ref)
