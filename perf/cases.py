"""The work a user of this framework has it do, as timed cases.

Every case goes through the package's public entry points the way a program
does: handles, weights and input fields are in hand (`prepare`), one `run` is
one pressure solve, one batch, one fractional step or one gradient of the
network.  Sizes come from the framework's workloads and tests; `draw` spreads
them over the whole range: 2D and 3D, powers of two and ragged sizes, every
solve mode a program chooses for itself, walls and periodic axes.

`exact` restates the mathematics in float64 torch, independently of the
package.
"""
import math
import os

import torch

import paper_1112_3507_gb300
from paper_1112_3507_gb300 import lowmach as lm
from paper_1112_3507_gb300.fractional import FractionalStep

GAMMA = 5.0 / 3.0
PER, WALL = lm.BC_PERIODIC, lm.BC_NEUMANN
WEIGHTS = os.path.join(os.path.dirname(paper_1112_3507_gb300.__file__), "weights", "unet_16_32_48_64.bin")
CHANNELS = (16, 32, 48, 64)          # of the network in WEIGHTS
EXACT_CELLS = 1 << 25                # larger solves have no float64 restatement within seconds
EXACT_STEPS = 4_000                  # conjugate-gradient steps of a float64 restatement, at most


# ---- the cases -------------------------------------------------------------------

def _solve(nx, ny, nz, mode="mixed", rtol=1e-8, ma=0.01, contrast=20.0, noise=0.01, wall_x=False):
    return dict(kind="solve", nx=nx, ny=ny, nz=nz, mode=mode, rtol=rtol, ma=ma, contrast=contrast, noise=noise,
                wall_x=wall_x)


def listed():
    return [
        # The smallest solve in earnest: a 2D test atmosphere at a tight tolerance, all latency.
        dict(_solve(64, 1, 64, rtol=1e-10, ma=0.1, contrast=31.6, noise=0.0), name="solve2d-64"),
        # A periodic axis with an odd count has no multigrid hierarchy: plain float64 conjugate gradients.
        dict(_solve(129, 1, 97, mode="jacobi", ma=0.1), name="jacobi2d-129x97"),
        # One time step of the Gresho vortex: explicit kernels around a warm-started solve.
        dict(kind="step", nx=256, ny=1, nz=256, ma=0.01, dt_factor=1.0, name="gresho2d-256"),
        # A held-out member of the training family, warm-started by the network.
        dict(_solve(256, 1, 256, mode="learned"), name="learned2d-256"),
        # A ragged 2D box between walls, off every tile size.
        dict(_solve(360, 1, 200, ma=0.03, contrast=10.0, wall_x=True), name="solve2d-360x200"),
        # Many uneven 2D problems at once, sides 128 to 1024 (a parameter study).
        dict(kind="batch", count=64, lo=128, hi=1024, pow2=True, spec=42, name="batch2d-64"),
        # A ragged 3D box: no axis is a multiple of 64.
        dict(_solve(120, 72, 88), name="solve3d-120x72x88"),
        # One fractional step in three dimensions at four times the acoustic step.
        dict(kind="step", nx=96, ny=96, nz=96, ma=0.05, dt_factor=4.0, name="step3d-96"),
        # The headline solve: 3D stratified convection.
        dict(_solve(256, 256, 256), name="solve3d-256"),
        # The largest solve: two orders below the acoustic Courant limit.
        dict(_solve(512, 512, 512, ma=0.001), name="solve3d-512"),
        # The paper's own discretization, Q1 finite elements.
        dict(kind="fe", nx=256, ny=256, nz=256, ma=0.01, rtol=1e-8, wall_x=False, name="fe3d-256"),
        # One gradient of the network's training loop at the trainer's batch.
        dict(kind="net", batch=16, height=256, width=256, backward=True, name="net-grad-16x256"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _extent(rng, lo, hi, odd=(1, 3, 5, 7, 9, 11, 13, 15), low2=3):
    """A cell count between lo and hi that halves at least `low2` times: odd * 2^k."""
    goal, best = _log(rng, lo, hi), None
    m = rng.choice(odd)
    for k in range(low2, 12):
        n = m << k
        if lo <= n <= hi and (best is None or abs(math.log(n / goal)) < abs(math.log(best / goal))):
            best = n
    return best or 1 << int(math.log2(goal))


def draw(rng):
    kind = rng.choice(("solve2", "solve2", "solve2", "solve3", "solve3", "solve3", "jacobi", "batch", "step", "step",
                       "fe", "net"))
    ma = _log(rng, 1e-3, 1e-1)
    contrast, wall_x = rng.uniform(5.0, 30.0), rng.random() < 0.3
    mode = "learned" if rng.random() < 0.25 else "mixed"
    if kind == "solve2":
        ma = max(ma, 4e-3)           # few halvings: below this a ragged box outlasts the largest listed solve
        return _solve(_extent(rng, 48, 2048), 1, _extent(rng, 48, 2048), mode=mode, rtol=rng.choice((1e-8, 1e-10)),
                      ma=ma, contrast=contrast, wall_x=wall_x)
    if kind == "solve3":
        if rng.random() < 0.3:
            n = (rng.choice((128, 256, 512)), rng.choice((64, 128, 256)), rng.choice((64, 128, 256)))
            mode = "mixed"
        else:
            n = (_extent(rng, 32, 224), _extent(rng, 32, 144), _extent(rng, 32, 144))
            ma = max(ma, 4e-3)
        return _solve(*n, mode=mode, ma=ma, contrast=contrast, wall_x=wall_x)
    if kind == "jacobi":
        three = rng.random() < 0.35
        return _solve(2 * rng.randint(16, 40 if three else 160) + 1, 2 * rng.randint(8, 24) + 1 if three else 1,
                      rng.randint(32, 96 if three else 200), mode="jacobi", ma=_log(rng, 1e-2, 1e-1),
                      contrast=contrast, wall_x=wall_x)
    if kind == "batch":
        return dict(kind="batch", count=int(_log(rng, 4, 64.9)), lo=64, hi=rng.choice((256, 512, 1024)),
                    pow2=rng.random() < 0.5, spec=rng.randint(0, 1 << 20))
    if kind == "step":
        three = rng.random() < 0.5
        hi = 128 if three else 1024
        return dict(kind="step", nx=_extent(rng, 32, hi), ny=_extent(rng, 32, 96) if three else 1,
                    nz=_extent(rng, 32, hi), ma=_log(rng, 1e-2, 1e-1), dt_factor=rng.choice((1.0, 2.0, 4.0)))
    if kind == "fe":
        three = rng.random() < 0.6
        return dict(kind="fe", nx=_extent(rng, 32, 144) if three else _extent(rng, 48, 640),
                    ny=_extent(rng, 32, 96) if three else 1,
                    nz=_extent(rng, 32, 96 if three else 512) + rng.choice((0, 0, 1)), ma=_log(rng, 1e-2, 1e-1),
                    rtol=1e-8, wall_x=wall_x)
    side = (64, 96, 128, 160, 200, 256, 320)
    return dict(kind="net", batch=int(_log(rng, 1, 24.9)), height=rng.choice(side), width=rng.choice(side),
                backward=rng.random() < 0.7)


# ---- inputs ----------------------------------------------------------------------

class _Field:
    """Seeded random fields of shape (nz, ny, nx) on the GPU."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)

    def uniform(self, shape):
        return 2.0 * torch.rand(shape, generator=self.gen, device="cuda", dtype=torch.float64) - 1.0

    def smooth(self, shape, bc, sigma=2.0):
        """White noise smoothed over `sigma` cells (wrapped or mirrored), zero mean, unit 2-norm."""
        w = torch.randn(shape, generator=self.gen, device="cuda", dtype=torch.float64)
        r = math.ceil(4 * sigma)
        taps = [math.exp(-0.5 * (t / sigma) ** 2) for t in range(-r, r + 1)]
        for axis, b in ((2, bc[0]), (1, bc[1]), (0, bc[2])):
            n = shape[axis]
            if n == 1:
                continue
            at, acc = torch.arange(n, device="cuda"), torch.zeros_like(w)
            for t, g in zip(range(-r, r + 1), taps):
                i = (at + t) % n if b == PER else (at + t) % (2 * n)
                if b != PER:
                    i = torch.where(i >= n, 2 * n - 1 - i, i)
                acc.add_(w.index_select(axis, i), alpha=g / sum(taps))
            w = acc
        w -= w.mean()
        return w / w.norm()


def _atmosphere(field, n, contrast, noise):
    """rho^n, rho^{n+1}, c_s^2 of a polytrope over one unit of height with seeded density noise."""
    nx, ny, nz = n
    z = (torch.arange(nz, device="cuda", dtype=torch.float64) + 0.5) / nz
    base = (1.0 - (1.0 - contrast ** (-2.0 / 3.0)) * z)[:, None, None]
    rho = (base ** 1.5 * (1.0 + noise * field.uniform((nz, ny, nx)))).contiguous()
    cs2 = (GAMMA * base ** 2.5 / rho).contiguous()
    rho_new = (rho * (1.0 + 0.1 * noise * field.uniform((nz, ny, nx)))).contiguous()
    return rho, rho_new, cs2


def _problem(c, seed):
    n = (c["nx"], c["ny"], c["nz"])
    bc = (WALL if c["wall_x"] else PER, PER, WALL)
    h = 1.0 / n[2]
    field = _Field(seed)
    rho, rho_new, cs2 = _atmosphere(field, n, c.get("contrast", 20.0), c.get("noise", 0.01))
    dt = 0.5 * h / (c["ma"] * float(cs2.max().sqrt()))
    f = field.smooth(rho.shape, bc)
    return dict(n=n, h=(h, h, h), bc=bc, rho=rho, rho_new=rho_new, cs2=cs2, dt=dt, f=f.contiguous())


def _batch_cases(c):
    import random
    rng = random.Random(c["spec"])
    sides = [s for s in (64, 128, 256, 512, 1024) if c["lo"] <= s <= c["hi"]]
    side = (lambda: rng.choice(sides)) if c["pow2"] else (lambda: _extent(rng, c["lo"], c["hi"], odd=(1, 3, 5)))
    return [_solve(side(), 1, side(), ma=_log(rng, 1e-3, 1e-1), contrast=rng.uniform(5.0, 30.0), noise=0.0)
            for _ in range(c["count"])]


def _vortex(c, seed):
    """The Gresho vortex (a column of it in 3D) on a periodic box, with seeded density noise."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    ma, h = c["ma"], (1.0 / nx, 1.0 / ny, 1.0 / nz)
    x = (torch.arange(nx, device="cuda", dtype=torch.float64) + 0.5) * h[0] - 0.5
    z = (torch.arange(nz, device="cuda", dtype=torch.float64) + 0.5) * h[2] - 0.5
    dx, dz = x[None, None, :].expand(nz, ny, nx), z[:, None, None].expand(nz, ny, nx)
    r = torch.sqrt(dx * dx + dz * dz)
    inner, ring = r <= 0.2, (r > 0.2) & (r <= 0.4)
    zero = torch.zeros_like(r)
    uphi = torch.where(inner, 5.0 * r, torch.where(ring, 2.0 - 5.0 * r, zero))
    p0 = 1.0 / (GAMMA * ma * ma)
    p = torch.where(inner, p0 + 12.5 * r * r,
                    torch.where(ring, p0 + 12.5 * r * r + 4.0 * (1.0 - 5.0 * r - math.log(0.2) + torch.log(r)),
                                zero + p0 - 2.0 + 4.0 * math.log(2.0)))
    rho = 1.0 + 0.01 * _Field(seed).uniform((nz, ny, nx))
    ux, uz = -dz / r * uphi, dx / r * uphi
    mom = torch.stack((rho * ux, 0.05 * rho, rho * uz) if ny > 1 else (rho * ux, zero, rho * uz))
    e = p / (GAMMA - 1.0) + 0.5 * (mom * mom).sum(0) / rho
    dt = c["dt_factor"] * 0.5 * min(h[0], h[2], h[1] if ny > 1 else 1.0) / float(
        (uphi + torch.sqrt(GAMMA * p / rho)).max())
    return dict(n=(nx, ny, nz), h=h, rho=rho.contiguous(), mom=mom.contiguous(), e=e.contiguous(), dt=dt)


def _images(c, seed):
    """Network inputs (v / rms, log rho, log of the acoustic number) and targets like the trainer's."""
    B, H, W = c["batch"], c["height"], c["width"]
    field = _Field(seed)
    x = torch.empty((B, H, W, 3), device="cuda")
    t = torch.empty((B, H, W), device="cuda")
    z = (torch.arange(H, device="cuda", dtype=torch.float64) + 0.5) / H
    for b in range(B):
        v = field.smooth((H, 1, W), (PER, PER, WALL)) * math.sqrt(H * W)
        rho = (1.0 - 0.8 * z)[:, None] ** 1.5 * (1.0 + 0.01 * field.uniform((H, W)))
        x[b, :, :, 0] = v.view(H, W)
        x[b, :, :, 1] = torch.log(rho / rho.mean())
        x[b, :, :, 2] = 0.1 * torch.log(3e3 / (1.0 - 0.8 * z))[:, None]
        t[b] = (field.smooth((H, 1, W), (PER, PER, WALL), sigma=6.0) * math.sqrt(H * W)).view(H, W)
    return x, t


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "solve":
        p = _problem(c, seed)
        g = lm.Grid(p["n"], p["h"], p["bc"])
        if c["mode"] == "learned":
            g.load_network(WEIGHTS)
        return dict(case=c, p=p, grid=g, x=torch.empty_like(p["f"]))
    if kind == "batch":
        ps = [_problem(s, seed * 1009 + k) for k, s in enumerate(_batch_cases(c))]
        return dict(case=c, ps=ps, grids=[lm.Grid(p["n"], p["h"], p["bc"]) for p in ps],
                    xs=[torch.empty_like(p["f"]) for p in ps])
    if kind == "step":
        v = _vortex(c, seed)
        return dict(case=c, v=v, sim=FractionalStep(v["n"], v["h"], (PER, PER, PER), GAMMA))
    if kind == "fe":
        p = _problem(dict(c, contrast=20.0, noise=0.01), seed)
        return dict(case=c, p=p, fe=lm.FEGrid(p["n"], p["h"], p["bc"]), b=torch.empty_like(p["f"]),
                    x=torch.empty_like(p["f"]))
    x, t = _images(c, seed)
    return dict(case=c, x=x, t=t, net=lm.Net.load(WEIGHTS), y=torch.empty_like(t), gy=torch.empty_like(t))


# ---- one pass --------------------------------------------------------------------

def run(s):
    c, kind = s["case"], s["case"]["kind"]
    if kind == "solve":
        p, g = s["p"], s["grid"]
        g.set_coefficients(p["rho"], p["rho_new"], p["cs2"], p["dt"])
        g.set_rhs(p["f"])
        g.solve(mode=c["mode"], rtol=c["rtol"])
        return g.solution(s["x"])
    if kind == "batch":
        ps = s["ps"]
        lm.batch_set_coefficients(s["grids"], [p["rho"] for p in ps], [p["rho_new"] for p in ps],
                                  [p["cs2"] for p in ps], [p["dt"] for p in ps])
        for g, p in zip(s["grids"], ps):
            g.set_rhs(p["f"])
        lm.batch_solve(s["grids"], rtol=1e-8)
        return [g.solution(x) for g, x in zip(s["grids"], s["xs"])]
    if kind == "step":
        v, sim = s["v"], s["sim"]
        sim.set_state(v["rho"], v["mom"], v["e"])
        sim.step(v["dt"])
        return dict(rho=sim.rho, mom=sim.mom, e=sim.e, p=sim.p)
    if kind == "fe":
        p, fe = s["p"], s["fe"]
        fe.set_state(p["rho"], p["rho_new"], p["cs2"], p["dt"])
        fe.mass_times(p["f"], s["b"])
        fe.solve(s["b"], s["x"], rtol=c["rtol"])
        return s["x"]
    net, (B, H, W) = s["net"], s["t"].shape
    net.forward(s["x"], s["y"], B, H, W)
    if not c["backward"]:
        return s["y"]
    net.mse(s["y"], s["t"], s["gy"], want_loss=False)
    net.backward(s["gy"])
    return dict(y=s["y"], grads=net.grads())


def work(case):
    """Each input and output once; a solve's arithmetic as one operator application, its least."""
    c, kind = case, case["kind"]
    if kind == "batch":
        cells = sum(s["nx"] * s["nz"] for s in _batch_cases(c))
        return {"bytes": 40.0 * cells, "flops": 13.0 * cells}
    if kind == "net":
        px = c["batch"] * c["height"] * c["width"]
        one, prev, ch = 0.0, 3, CHANNELS
        for l in range(4):
            one += 18.0 * (prev * ch[l] + ch[l] * ch[l]) / 4 ** l
            prev = ch[l]
            if l < 3:
                one += 18.0 * ((ch[l] + ch[l + 1]) * ch[l] + ch[l] * ch[l]) / 4 ** l
        return {"bytes": 16.0 * px + (4.0 * px if c["backward"] else 0.0),
                "flops": (3.0 if c["backward"] else 1.0) * one * px}
    cells = c["nx"] * c["ny"] * c["nz"]
    if kind == "step":
        return {"bytes": 88.0 * cells, "flops": 300.0 * cells}
    return {"bytes": 40.0 * cells, "flops": (60.0 if kind == "fe" else 13.0) * cells}


# ---- float64 restatements --------------------------------------------------------

AXES = ((2, 0), (1, 1), (0, 2))      # (tensor axis, grid axis)


def _cg(apply, diag, f):
    """Jacobi-preconditioned conjugate gradients to the float64 floor."""
    x, r = torch.zeros_like(f), f.clone()
    z = r / diag
    p, rz, goal = z.clone(), torch.sum(r * z), 1e-15 * float(f.norm())
    for k in range(EXACT_STEPS):
        q = apply(p)
        a = rz / torch.sum(p * q)
        x += a * p
        r -= a * q
        if k % 50 == 49 and not float(r.norm()) > goal:
            break
        z = r / diag
        new = torch.sum(r * z)
        p = z + (new / rz) * p
        rz = new
    return x


def _poisson(rho_old, rho_new, cs2, dt, h, bc):
    """(apply, diagonal) of c~ x - div(grad x / rho) in finite volumes."""
    c = 1.0 / (dt * dt * rho_old * cs2)
    faces = []
    for ax, a in AXES:
        if c.shape[ax] > 1:
            g = 2.0 / ((rho_new + rho_new.roll(1, ax)) * h[a] ** 2)
            if bc[a] == WALL:
                g.narrow(ax, 0, 1).zero_()
            faces.append((ax, g))
    diag = c.clone()
    for ax, g in faces:
        diag += g + g.roll(-1, ax)

    def apply(x):
        y = c * x
        for ax, g in faces:
            flux = g * (x - x.roll(1, ax))
            y += flux
            y -= flux.roll(-1, ax)
        return y

    return apply, diag


def _exact_problem(c, seed):
    if c["nx"] * c["ny"] * c["nz"] > EXACT_CELLS:
        return None
    p = _problem(c, seed)
    return _cg(*_poisson(p["rho"], p["rho_new"], p["cs2"], p["dt"], p["h"], p["bc"]), p["f"])


def _exact_fe(c, seed):
    if c["nx"] * c["ny"] * c["nz"] > 3_000_000:
        return None
    p = _problem(dict(c, contrast=20.0, noise=0.01), seed)
    shape, h, bc = p["f"].shape, p["h"], p["bc"]
    live = [(ax, a) for ax, a in AXES if shape[ax] > 1]
    vol = torch.ones(shape, device="cuda", dtype=torch.float64)
    kappa, corners = None, [()]
    for ax, a in live:
        corners = [o + (b,) for o in corners for b in (0, 1)]
        w = torch.full((shape[ax],), h[a], device="cuda", dtype=torch.float64)
        if bc[a] == WALL:
            w[0] = w[-1] = 0.5 * h[a]
        vol = vol * w.view([-1 if k == ax else 1 for k in range(3)])
    axes = [ax for ax, _ in live]
    kappa = len(corners) / sum(p["rho_new"].roll([-b for b in o], axes) for o in corners)
    for ax, a in live:
        if bc[a] == WALL:
            kappa.narrow(ax, shape[ax] - 1, 1).zero_()
    hs = [h[a] for _, a in live]

    def entry(o, q):
        """The reference element's stiffness between corners o and q."""
        total = 0.0
        for d in range(len(hs)):
            term = 1.0
            for e in range(len(hs)):
                same = o[e] == q[e]
                term *= (1.0 if same else -1.0) / hs[e] if e == d else hs[e] * (2.0 if same else 1.0) / 6.0
            total += term
        return total

    mass = vol / (p["dt"] ** 2 * p["rho"] * p["cs2"])

    def apply(x):
        at = [x.roll([-b for b in o], axes) for o in corners]
        y = mass * x
        for o in corners:
            t = sum(entry(o, q) * xq for q, xq in zip(corners, at))
            y += (kappa * t).roll(list(o), axes)
        return y

    diag = mass + entry(corners[0], corners[0]) * sum(kappa.roll(list(o), axes) for o in corners)
    return _cg(apply, diag, vol * p["f"])


def _exact_step(c, seed):
    v = _vortex(c, seed)
    h, dt, rho, mom, e = v["h"], v["dt"], v["rho"], v["mom"], v["e"]
    live = [(ax, a) for ax, a in AXES if rho.shape[ax] > 1]
    p = (GAMMA - 1.0) * (e - 0.5 * (mom * mom).sum(0) / rho)
    cs2 = GAMMA * p / rho
    new = []
    for q in (rho, mom[0], mom[1], mom[2], e):       # advection: upwind minmod-limited fluxes
        out = q.clone()
        for ax, a in live:
            u = (mom[a] + mom[a].roll(1, ax)) / (rho + rho.roll(1, ax))
            lo, hi = q - q.roll(1, ax), q.roll(-1, ax) - q
            s = torch.where(lo * hi > 0, torch.where(lo.abs() < hi.abs(), lo, hi), torch.zeros_like(q))
            flux = u * torch.where(u > 0, (q + 0.5 * s).roll(1, ax), q - 0.5 * s)
            out -= dt * (flux.roll(-1, ax) - flux) / h[a]
        new.append(out)
    rho1, mom_s, e_s = new[0], torch.stack(new[1:4]), new[4]

    def grad(P, r, ax, a):
        face = (P * r.roll(1, ax) + P.roll(1, ax) * r) / (r + r.roll(1, ax))
        return (face.roll(-1, ax) - face) / h[a]

    f, us = p.clone(), {}
    for ax, a in live:
        f -= dt * mom[a] / rho * grad(p, rho, ax, a)
    f /= dt * dt * rho * cs2
    for ax, a in live:
        us[a] = (mom_s[a] + mom_s[a].roll(1, ax)) / (rho1 + rho1.roll(1, ax))
        f -= (us[a].roll(-1, ax) - us[a]) / (h[a] * dt)
    bc = (PER, PER, PER)
    op, diag = _poisson(rho, rho1, cs2, dt, h, bc)
    x = p + _cg(op, diag, f - op(p))
    mom1, div, ugp = mom_s.clone(), torch.zeros_like(x), torch.zeros_like(x)
    for ax, a in live:
        g = grad(x, rho1, ax, a)
        mom1[a] -= dt * g
        u1 = us[a] - dt * (x - x.roll(1, ax)) / h[a] * 2.0 / (rho1 + rho1.roll(1, ax))
        div += (u1.roll(-1, ax) - u1) / h[a]
        ugp += mom1[a] / rho1 * g
    e1 = e_s - dt * (x * div + ugp)
    p1 = (GAMMA - 1.0) * (e1 - 0.5 * (mom1 * mom1).sum(0) / rho1)
    return dict(rho=rho1.reshape(-1), mom=mom1.reshape(-1), e=e1.reshape(-1), p=p1.reshape(-1))


def _exact_net(c, seed):
    F = torch.nn.functional
    x, t = _images(c, seed)
    net = lm.Net.load(WEIGHTS)
    flat = torch.as_tensor(net.params(), device="cuda").double().requires_grad_(c["backward"])
    net.close()
    at = 0

    def take(*shape):
        nonlocal at
        n = math.prod(shape)
        at += n
        return flat[at - n:at].view(shape)

    ch = CHANNELS
    shapes = [(a, b) for l in range(4) for a, b in ((3 if l == 0 else ch[l - 1], ch[l]), (ch[l], ch[l]))]
    shapes += [(a, b) for l in (2, 1, 0) for a, b in ((ch[l + 1] + ch[l], ch[l]), (ch[l], ch[l]))]
    layers = iter([(take(3, 3, a, b).permute(3, 2, 0, 1), take(b)) for a, b in shapes])
    last = take(ch[0]), take(1)

    def two(v):
        for w, b in (next(layers), next(layers)):
            v = F.relu(F.conv2d(v, w, b, padding=1))
        return v

    v, skips = x.double().permute(0, 3, 1, 2), []
    for l in range(4):
        v = two(v if l == 0 else F.avg_pool2d(v, 2))
        skips.append(v)
    for l in (2, 1, 0):
        v = two(torch.cat((F.interpolate(v, scale_factor=2, mode="nearest"), skips[l]), 1))
    y = torch.einsum("bchw,c->bhw", v, last[0]) + last[1]
    if not c["backward"]:
        return y
    F.mse_loss(y, t.double()).backward()
    return dict(y=y.detach(), grads=flat.grad)


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        return _exact_problem(case, seed)
    if kind == "batch":
        return [_exact_problem(s, seed * 1009 + k) if s["nx"] * s["nz"] <= 1 << 16 else None
                for k, s in enumerate(_batch_cases(case))]
    if kind == "fe":
        return _exact_fe(case, seed)
    return _exact_step(case, seed) if kind == "step" else _exact_net(case, seed)
