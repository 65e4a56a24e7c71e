"""Integer stencil sums beside walls: a neighbour of no weight, whatever its size,
leaves the row's accuracy alone (arithmetic on the host; the solvers' refinement
residuals on the device); and rows whose classes of neighbours have factors of
their own, as finite elements of unequal sides have."""
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
#include "lm_intfp.cuh"
static uint64_t bits(double d) { uint64_t u; memcpy(&u, &d, 8); return u; }
static double value(uint64_t u) { double d; memcpy(&d, &u, 8); return d; }
int main() {
    std::mt19937_64 g(11);
    const uint64_t M = (1ull << 52) - 1;
    long bad = 0, taken = 0;
    for (long i = 0; i < 1000000; ++i) {
        const bool wide = i & 1;                 // weights within a factor of two, the x of any spread
        double x[7], w[6];
        lm::ExpRange rx, rw;
        const int p0 = (int)(g() % 400) - 200, q0 = (int)(g() % 400) - 200;
        auto mant = [&] { return value((g() & M) | 1023ull << 52); };
        for (int o = 0; o < 7; ++o)
            x[o] = ldexp(mant(), p0 + (int)(wide ? g() % 60 : g() % 6)) * (g() & 1 ? -1 : 1);
        for (int o = 0; o < 6; ++o) {
            w[o] = ldexp(mant(), q0 + (int)(wide ? 0 : g() % 5));
            if (g() % 3 == 0) w[o] = 0.0, x[o] = ldexp(x[o], (int)(g() % 300) - 100);
        }
        uint64_t xu[7], wu[6];
        xu[6] = bits(x[6]);
        rx.add((uint32_t)(xu[6] >> 32) & 0x7fffffffu);
        for (int o = 0; o < 6; ++o) {
            wu[o] = bits(w[o]);
            xu[o] = lm::fix_live(bits(x[o]), wu[o], xu[6]);
            rx.add((uint32_t)(xu[o] >> 32) & 0x7fffffffu), rw.add((uint32_t)(wu[o] >> 32));
        }
        if (!lm::fix_ok(rx, 5, rw, 4)) continue;
        ++taken;
        const lm::Limbs c = lm::fix<5>(xu[6], rx.top());
        lm::FixSum s;
        long double S = 0, mag = 0;
        for (int o = 0; o < 6; ++o) {
            s.mac(lm::fix_diff<5>(c, xu[o], rx.top()), lm::fix_abs<4>(wu[o], rw.top()));
            const long double t = (long double)w[o] * ((long double)x[6] - x[o]);
            if (w[o] != 0) S += t, mag += fabsl(t);
        }
        const double got = value(lm::fix_round(s.total(), lm::fix_scale<5, 4>(rx.top(), rw.top())));
        bad += !(fabsl(got - S) <= ldexpl(mag, -52));
    }
    const uint64_t inf = 0x7ffull << 52, one = bits(1.0);
    bad += lm::fix_live(inf, 0, one) != inf || lm::fix_live(inf + 1, 1ull << 63, one) != inf + 1;
    bad += lm::fix_live(0, 0, one) != one || lm::fix_live(7, 1, one) != 7;
    printf("%ld of %ld\n", bad, taken);
    return bad != 0 || taken < 400000;
}
"""


CLASSES = r"""
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include "lm_intfp.cuh"
static uint64_t bits(double d) { uint64_t u; memcpy(&u, &d, 8); return u; }
static double value(uint64_t u) { double d; memcpy(&d, &u, 8); return d; }
int main() {
    std::mt19937_64 g(13);
    double ei = 0, ef = 0, mi = 0, mf = 0;
    long n = 0;
    for (long i = 0; i < 1500000; ++i) {         // three classes of four neighbours, factors 2^-12 to 2
        double x[13], w[12], c[3];
        auto mant = [&] { return value((g() & ((1ull << 52) - 1)) | 1023ull << 52); };
        const int spread = 6 + (int)(g() % 50);
        for (int o = 0; o < 13; ++o) {           // any spread, or one class far above the rest
            const int e = i % 4 ? (int)(g() % spread) : o < 4 && g() % 4 == 0 ? spread : (int)(g() % 4);
            x[o] = ldexp(mant(), e) * (g() & 1 ? -1 : 1);
        }
        for (int o = 0; o < 12; ++o) w[o] = mant();
        for (int q = 0; q < 3; ++q) c[q] = ldexp(mant(), -(int)(g() % 12));
        const double cm = std::max(c[0], std::max(c[1], c[2]));
        lm::ExpRange rx, rw, rs;
        auto h = [](double v) { return (uint32_t)(bits(v) >> 32) & 0x7fffffffu; };
        for (int o = 0; o < 13; ++o) {
            rx.add(h(x[o]));
            if (o == 12 || 4.0 * c[o / 4] >= cm) rs.add(h(x[o]));
        }
        for (int o = 0; o < 12; ++o) rw.add(h(w[o]));
        if (rx.spread() <= 5 || !lm::fix_ok(rx, 5, rw, 3, rs)) continue;
        const lm::Limbs cc = lm::fix<5>(bits(x[12]), rx.top());
        double yi = 0, yf = 0;
        long double S = 0, mag = 0;
        for (int q = 0; q < 3; ++q) {
            lm::FixSum s;
            double a = 0;
            for (int o = 4 * q; o < 4 * q + 4; ++o) {
                s.mac(lm::fix_diff<5>(cc, bits(x[o]), rx.top()), lm::fix_abs<3>(bits(w[o]), rw.top()));
                a = fma(w[o], x[12] - x[o], a);
                const long double t = (long double)c[q] * w[o] * ((long double)x[12] - x[o]);
                S += t, mag += fabsl(t);
            }
            yi = fma(c[q], value(lm::fix_round(s.total(), lm::fix_scale<5, 3>(rx.top(), rw.top()))), yi);
            yf = fma(c[q], a, yf);
        }
        const double a = fabsl(yi - S) / mag, b = fabsl(yf - S) / mag;
        ei += a, ef += b, ++n;
        mi = std::max(mi, a), mf = std::max(mf, b);
    }
    printf("%ld rows: mean %g against %g, largest %g against %g\n", n, ei / n, ef / n, mi, mf);
    return !(n > 500000 && ei <= ef && mi <= mf);
}
"""


# The rows that the integer form takes are as close to the exact sum as the float64
# form's, on average and at worst.
@pytest.mark.parametrize("program", [PROGRAM, CLASSES], ids=["walls", "classes"])
def test_rows_on_the_host(tmp_path, program):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "q.cpp", tmp_path / "q"
    src.write_text(program)
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout


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


# The half of the cells at the far wall holds values 2^30 times the other's, with
# coefficients of 2^-48: its rows, rounding included, are small beside the near
# half's, whose first rows the indexing joins to the far wall by a face of no
# weight.  Only the rounding of each row's terms is left, (terms + 2) half units.
@pytest.mark.gpu
@pytest.mark.parametrize("n", [(40, 1, 38), (34, 10, 12), (12, 36, 10)])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("h", [(1 / 32, 1 / 32, 1 / 32), (0.1, 0.2, 0.15)])
def test_residuals_beside_walls(lm, n, axis, h):
    import torch
    if n[axis] == 1:
        pytest.skip("one cell")
    rng = np.random.default_rng(n[0] + axis)
    N = n[0] * n[1] * n[2]
    shape = (n[2], n[1], n[0])
    bc = tuple(1 if a == axis else 0 for a in range(3))
    far = np.broadcast_to((np.arange(n[axis]) >= n[axis] // 2).reshape([-1 if a == 2 - axis else 1 for a in range(3)]),
                          shape)
    x = np.where(far, 2.0 ** 30, 1.0) * (1.0 + rng.random(shape))
    rho = np.where(far, 2.0 ** 48, 1.0)
    ct = np.where(far, 2.0 ** -48, 1.0) * (1.0 + rng.random(shape))
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a).ravel(), device="cuda")
    tol = lambda mag, terms, f: 2 * (terms + 2) * 2.0 ** -53 * np.linalg.norm(mag) / np.linalg.norm(f)
    with lm.Grid(n, h, bc) as g:
        g.set_coefficients_raw(ct.ravel(), rho.ravel())
        f = d(np.empty(N))
        g.apply(d(x), f)
        g.set_rhs(f)
        g.set_initial_guess(d(x))
        rel = g.solve(rtol=1.0, use_x0=1)["rel_residual"]
        c, *gs = (t.cpu().numpy().reshape(shape) for t in g.coefficients())
    mag = np.abs(c * x)
    for a, gm in enumerate(gs):
        t = gm * np.abs(x - np.roll(x, 1, 2 - a))
        mag += t + np.roll(t, -1, 2 - a)
    assert rel <= tol(mag, 7, f.cpu().numpy())
    from oracle import fem as F
    op = F.FEOperator(ct, rho, h, bc)
    with lm.FEGrid(n, h, bc) as fe:
        fe.set_coefficients(ct.ravel(), rho.ravel())
        fe.apply(d(x), f)
        rel = fe.solve(f, d(x), rtol=1.0, use_x0=1)["rel_residual"]
    mag = np.abs(op.volume * op.ct * x)
    xc = [op._corner(x, c) for c in op.corners]
    for p in range(len(op.corners)):
        for q in range(len(op.corners)):
            mag += op._back(op.kappa_e * abs(op.kref[p, q]) * np.abs(xc[q] - xc[p]), op.corners[p])
    assert rel <= tol(mag, 27, f.cpu().numpy())
