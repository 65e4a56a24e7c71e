"""Float64 quotients and stencil sums on the integer pipe: their arithmetic compiled
for the host and compared with the hardware division and with integers, and the
device's own through the entry points that use it."""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1112_3507_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>
#include "lm_intfp.cuh"
static uint64_t bits(double d) { uint64_t u; memcpy(&u, &d, 8); return u; }
static double value(uint64_t u) { double d; memcpy(&d, &u, 8); return d; }
// the device's idiv for normal operands, its seed off by `off` units
static double quotient(double a, double b, int off) {
    const uint64_t M = (1ull << 52) - 1, ua = bits(a), ub = bits(b), mb = ub & M;
    const uint32_t fb = 0x3f800000u | (uint32_t)(mb >> 29);
    float f, r;
    memcpy(&f, &fb, 4);
    r = 1.0f / f;
    uint32_t rb;
    memcpy(&rb, &r, 4);
    if (rb + off <= 0x3f800000u && rb + off >= 0x3f000000u) rb += off;
    const int e = (int)(ua >> 52 & 0x7ff) - (int)(ub >> 52 & 0x7ff) + 1023;
    const int64_t q = lm::idiv_core(ua & M, mb, e, lm::idiv_recip(mb | (1ull << 52), rb));
    return value((uint64_t)q | ((ua ^ ub) & (1ull << 63)));
}
int main() {
    std::mt19937_64 g(7);
    const uint64_t M = (1ull << 52) - 1, one = 1023ull << 52;
    std::vector<uint64_t> c;
    for (int i = 0; i < 8; ++i) c.push_back(i), c.push_back(M - i);
    for (int b = 0; b < 52; ++b)
        for (int d = -1; d <= 1; ++d) c.push_back(((1ull << b) + d) & M), c.push_back((M - (1ull << b) + d) & M);
    for (int i = 0; i < 40; ++i) c.push_back(g() & M);
    long bad = 0;
    for (uint64_t a : c)
        for (uint64_t b : c)
            for (int off = -2; off <= 2; ++off)
                bad += quotient(value(one | a), value(one | b), off) != value(one | a) / value(one | b);
    for (long i = 0; i < 3000000; ++i) {
        const double a = value((g() & M) | ((uint64_t)(600 + g() % 800) << 52)) * (i & 1 ? -1 : 1);
        const double b = value((g() & M) | ((uint64_t)(600 + g() % 800) << 52));
        bad += quotient(a, b, (int)(i % 5) - 2) != a / b;
    }
    // minmod over all magnitudes, signs, zeros, subnormals, infinities and NaN
    for (long i = 0; i < 1000000; ++i) {
        auto any = [&] {
            const int e = i % 3 == 0 ? g() % 2048 : i % 3 == 1 ? 480 + g() % 64 : (g() & 1 ? 0 : 1020 + g() % 60);
            const uint64_t m = g() % 5 == 0 ? 0 : g() % 5 == 0 ? 1 : g() & M;
            return (uint64_t)e << 52 | m | (g() & 1) << 63;
        };
        const uint64_t u = any(), v = g() % 16 == 0 ? u : any();
        const double a = value(u), b = value(v);
        bad += lm::minmod_bits(u, v) != bits(a * b > 0.0 ? (fabs(a) < fabs(b) ? a : b) : 0.0);
    }
    // sums of products of differences, against integers: mantissas A, B of 53 bits,
    // x = +-A 2^p with p < 6, w = B 2^q with q < 5, or zero
    for (long i = 0; i < 300000; ++i) {
        const int mode = i % 4, p0 = (int)(g() % 1200) - 600, q0 = (int)(g() % 600) - 300;
        int64_t X[7], W[6];
        uint64_t xu[7], wu[6];
        lm::ExpRange rx, rw;
        auto mant = [&] { return (int64_t)(mode == 0 ? M - (g() & 3) : mode == 1 ? g() & 3 : g() & M) | (1ll << 52); };
        for (int o = 0; o < 7; ++o) {
            const int64_t p = mode == 3 ? 5 : g() % 6, a = g() % 11 ? mant() : 0;
            X[o] = g() & 1 && mode != 3 ? -(a << p) : a << p;
            xu[o] = a ? ((uint64_t)(p0 + p + 1075) << 52 | (a & M)) | (X[o] < 0 ? 1ull << 63 : 0) : 0;
            rx.add((uint32_t)(xu[o] >> 32) & 0x7fffffffu);
        }
        for (int o = 0; o < 6; ++o) {
            const int64_t q = g() % 5, b = g() % 7 ? mant() : 0;
            W[o] = b << q;
            wu[o] = b ? (uint64_t)(q0 + q + 1075) << 52 | (b & M) : 0;
            rw.add((uint32_t)(wu[o] >> 32));
        }
        if (!lm::fix_ok(rx, 5, rw, 4)) continue;
        const lm::Limbs c = lm::fix<5>(xu[6], rx.top());
        lm::FixSum s;
        __int128 S = 0;
        for (int o = 0; o < 6; ++o) {
            s.mac(lm::fix_diff<5>(c, xu[o], rx.top()), lm::fix_abs<4>(wu[o], rw.top()));
            S += (__int128)(X[6] - X[o]) * W[o];
        }
        const uint64_t e = lm::fix_scale<5, 4>(rx.top(), rw.top());
        bad += value(lm::fix_round(s.total(), (int)e)) != ldexp((double)S, p0 + q0);
    }
    printf("%ld\n", bad);
    return bad != 0;
}
"""


def test_arithmetic_on_the_host(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "q.cpp", tmp_path / "q"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout


def _wide(rng, n, lo, hi):
    """Positive values of random mantissas (corners among them) and exponents lo .. hi - 1."""
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    k = rng.integers(0, 52, n // 4).astype(np.uint64)
    m[: n // 4] = (np.uint64(1) << k) - rng.integers(0, 2, n // 4).astype(np.uint64)
    m[n // 4: n // 2] = (np.uint64((1 << 52) - 1)) - m[: n // 4]
    e = (rng.integers(lo, hi, n) + 1023).astype(np.uint64)
    return ((e << np.uint64(52)) | m).view(np.float64)


@pytest.fixture(scope="module")
def lm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1112_3507_gb300 import build as B
    if not os.path.exists(B.LIB) or any(os.path.getmtime(s) > os.path.getmtime(B.LIB) for s in B.sources()):
        B.build()
    from paper_1112_3507_gb300 import lowmach
    return lowmach


@pytest.mark.gpu
@pytest.mark.parametrize("lo,hi", [(-8, 8), (-500, 500), (-1022, -900), (900, 1023)])
def test_quotient_on_the_device(lm, lo, hi):
    """c_s^2 = (gamma p) / rho of the ideal-gas reset, bit by bit, to the ends of the normal range and past them."""
    import torch
    rng = np.random.default_rng(abs(hi))
    n, gamma = 1 << 20, 1.5
    rho, e = _wide(rng, n, lo, hi), _wide(rng, n, -300, 300)
    e[:6] = [-0.0, 5e-324, 1e308, np.inf, np.nan, 2.0 ** -1022]
    e[12:4096] = 0.0
    rho[6:12] = [0.0, 5e-324, 2.0 ** -1022, np.inf, np.nan, 1.7e308]
    d = lambda a: torch.as_tensor(a, device="cuda")
    p, cs2 = d(np.empty(n)), d(np.empty(n))
    lm.eos_ideal(gamma, d(rho), d(np.zeros(3 * n)), d(e), p, cs2)
    p, cs2 = p.cpu().numpy(), cs2.cpu().numpy()
    with np.errstate(all="ignore"):
        want = (gamma * p) / rho
    assert np.array_equal(cs2.view(np.int64)[~np.isnan(want)], want.view(np.int64)[~np.isnan(want)])
    assert np.array_equal(np.isnan(cs2), np.isnan(want))


@pytest.mark.gpu
@pytest.mark.parametrize("h", [1.0 / 64, 1.0 / 48])
def test_assembly_bits(lm, h):
    """Reciprocals, the scaling by 2/h^2 and the float32 copies of an assembly, bit by bit."""
    import torch
    rng = np.random.default_rng(5)
    n = (64, 32, 16)
    N = n[0] * n[1] * n[2]
    ro, rn, c2 = _wide(rng, N, -20, 10), _wide(rng, N, -30, 20), _wide(rng, N, -40, 40)
    dt = 0.37
    g = lm.Grid(n, (h, h, h), (0, 0, 1))
    g.set_coefficients(ro, rn, c2, dt)
    ct, gx, gy, gz = (t.cpu().numpy() for t in g.coefficients())
    assert np.array_equal(ct, 1.0 / ((dt * dt) * ro * c2))
    r = rn.reshape(n[2], n[1], n[0])
    for axis, got in ((2, gx), (1, gy), (0, gz)):
        want = (2.0 / (h * h)) * (1.0 / (r + np.roll(r, 1, axis)))
        if axis == 0:
            want[0] = 0.0
        assert np.array_equal(got, want.ravel())
    import ctypes
    c32, r32 = torch.empty(N, device="cuda"), torch.empty(N, device="cuda")
    scale = ctypes.c_double()
    P = lambda t: ctypes.c_void_p(t.data_ptr())
    assert lm.lib().lm_mg_level_coefficients(g._g, 0, P(c32), P(r32), ctypes.byref(scale), None) == 0
    torch.cuda.synchronize()
    assert np.array_equal(c32.cpu().numpy(), ct.astype(np.float32))
    assert np.array_equal(r32.cpu().numpy() * np.float32(scale.value), rn.astype(np.float32))
    g.close()


def _field(kind, N, rng):
    if kind == "near one":
        return 1.0 + 1e-6 * rng.standard_normal(N)
    if kind == "both signs":
        return rng.standard_normal(N) * 1e-30
    x = rng.standard_normal(N) * 2.0 ** rng.integers(-40, 40, N)      # wide
    x[rng.random(N) < 0.2] = 0.0
    return x


@pytest.mark.gpu
@pytest.mark.parametrize("n,h", [((40, 1, 37), (1 / 32, 1.0, 1 / 32)), ((34, 10, 12), (0.1, 0.2, 0.15)), ((64, 24, 32), (1 / 64,) * 3)])
@pytest.mark.parametrize("kind", ["near one", "both signs", "wide"])
@pytest.mark.parametrize("spread", [0.05, 3.0])
def test_refinement_residuals(lm, n, h, kind, spread):
    """f - A x of the solvers' refinement where f is A x from the float64 apply: only
    the rounding of the row's terms is left, (terms + 2) half units of their sum each."""
    import torch
    rng = np.random.default_rng(n[0])
    N = n[0] * n[1] * n[2]
    shape = (n[2], n[1], n[0])
    rho = np.exp(rng.uniform(-spread, spread, N))
    ct = np.exp(rng.uniform(-1.0, 1.0, N))
    x = _field(kind, N, rng)
    bc = (0, 0, 1)
    d = lambda a: torch.as_tensor(a, device="cuda")
    ndim = 2 if n[1] == 1 else 3
    with lm.Grid(n, h, bc) as g:
        g.set_coefficients_raw(ct, rho)
        f = d(np.empty(N))
        g.apply(d(x), f)
        g.set_rhs(f)
        g.set_initial_guess(d(x))
        rel = g.solve(rtol=1.0, use_x0=1)["rel_residual"]
        c, *gs = (t.cpu().numpy().reshape(shape) for t in g.coefficients())
    xs = x.reshape(shape)
    mag = np.abs(c * xs)
    for a, gm in enumerate(gs):
        t = gm * np.abs(xs - np.roll(xs, 1, 2 - a))
        mag += t + np.roll(t, -1, 2 - a)
    tol = lambda mag, terms, f: 2 * (terms + 2) * 2.0 ** -53 * np.linalg.norm(mag) / np.linalg.norm(f)
    assert rel <= tol(mag, 7, f.cpu().numpy())
    from oracle import fem as F
    op = F.FEOperator(ct.reshape(shape), rho.reshape(shape), h, bc)
    with lm.FEGrid(n, h, bc) as fe:
        fe.set_coefficients(ct, rho)
        fe.apply(d(x), f)
        rel = fe.solve(f, d(x), rtol=1.0, use_x0=1)["rel_residual"]
    mag = np.abs(op.volume * op.ct * xs)
    xc = [op._corner(xs, c) for c in op.corners]
    for p in range(len(op.corners)):
        for q in range(len(op.corners)):
            mag += op._back(op.kappa_e * abs(op.kref[p, q]) * np.abs(xc[q] - xc[p]), op.corners[p])
    assert rel <= tol(mag, 27, f.cpu().numpy())
