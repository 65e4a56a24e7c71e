"""The integer-pipe float64 quotient: its arithmetic compiled for the host and
compared with the hardware division, and the device's own through the entry
points that use it."""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1112_3507_gb300", "csrc")

PROGRAM = r"""
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
    printf("%ld\n", bad);
    return bad != 0;
}
"""


def test_quotient_on_the_host(tmp_path):
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
