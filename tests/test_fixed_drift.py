"""The fixed-point Kepler solver (csrc/whg_fixed.cuh) on the CPU: its host build
against the drift's Lagrange coefficients in 113-bit arithmetic, and the
inputs it must leave to the FP64 solver."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#include "whg_fixed.cuh"
#if defined(__aarch64__)
typedef long double Q;
#else
typedef __float128 Q;
#endif
static Q root(Q x) { Q y = sqrt((double)x); for (int i = 0; i < 4; ++i) y = (y + x / y) / 2; return y; }
extern "C" int fixed_solve(int T, double mu, double h, double r0sq, double eta0, double v2, double* out)
{
    whg::fixed::Solution o{};
    const bool ok = T == 8 ? whg::fixed::solve<8, true>(mu, h, r0sq, eta0, v2, o)
                           : whg::fixed::solve<6, true>(mu, h, r0sq, eta0, v2, o);
    const double v[9] = {o.fm1n, o.g, o.fdn, o.gdm1n, o.s, o.g1, o.g2, o.g3, o.Ri};
    for (int i = 0; i < 9; ++i) out[i] = v[i];
    return ok;
}
// The same nine values relative errors (1 - computed/exact; g1.. as they are),
// the map's own series length T and Newton steps to convergence.
extern "C" void errors(int T, double mu, double h, double r0sq, double eta0, double v2, const double* c, double* err)
{
    const Q r0 = root(r0sq), w = (Q)h / r0, a = eta0 * w / r0, m = mu / r0 * w * w, V = v2 * w * w;
    const Q B = 2 * m - V, b = V - m;
    Q s = 1, g0, g1, g2, g3, R;
    for (int it = 0;; ++it) {
        const Q z = B * s * s;
        Q c2 = 0, c3 = 0, t2 = Q(1) / 2, t3 = Q(1) / 6;
        for (int k = 0; k <= T; ++k) {
            c2 += t2; c3 += t3;
            t2 *= -z / ((2 * k + 3) * (2 * k + 4));
            t3 *= -z / ((2 * k + 4) * (2 * k + 5));
        }
        g2 = s * s * c2; g3 = s * s * s * c3; g1 = s - B * g3; g0 = 1 - B * g2;
        R = 1 + a * g1 + b * g2;
        if (it == 14) break;
        s -= (s - 1 + a * g2 + b * g3) / R;
    }
    const Q x[9] = {m * g2, h * (1 - m * g3), mu / r0 * w / r0 * g1 / R, m * g2 / R, s, g1, g2, g3, 1 / R};
    for (int i = 0; i < 9; ++i) err[i] = (double)((c[i] - x[i]) / x[i]);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-O1", "-std=gnu++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2307_05683_gb300", "csrc"), str(src), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    D, P = ctypes.c_double, ctypes.c_void_p
    lib.fixed_solve.argtypes = [ctypes.c_int, D, D, D, D, D, P]
    lib.errors.argtypes = [ctypes.c_int, D, D, D, D, D, P, P]
    return lib


def _orbit(rng, e, frac, a=None, mu=None):
    """r0^2, eta0, v^2 at a random phase of an (a, e) orbit, h = frac of its period."""
    mu = 10.0 ** rng.uniform(-1, 1) if mu is None else mu
    a = 10.0 ** rng.uniform(-2, 3) if a is None else a
    E = rng.uniform(-np.pi, np.pi)
    r = a * (1 - e * np.cos(E))
    return (mu, 2 * np.pi * np.sqrt(a ** 3 / mu) * frac, r * r, e * np.sqrt(mu * a) * np.sin(E),
            mu * (2 / r - 1 / a))


@pytest.mark.parametrize("T", [6, 8])
@pytest.mark.parametrize("e,frac", [((0.0, 0.0), (0.05, 0.05)), ((0.0, 0.3), (0.02, 0.1)), ((0.0, 0.05), (0.1, 0.16)),
                                    ((0.3, 0.6), (0.005, 0.06)), ((0.0, 0.1), (1e-9, 1e-3)), ((0.6, 0.9), (1e-4, 0.004))])
def test_coefficients_against_113_bits(lib, T, e, frac):
    """Every output is one double rounded from a value of at least 55 correct
    bits: within 2^-53 of its size for the rounding and 2^-55 for the rest
    (sums of a few products, each wrong by 2^-60 of order one to 2^-57)."""
    rng = np.random.default_rng(11)
    out, err = np.zeros(9), np.zeros(9)
    worst = np.zeros(9)
    for _ in range(1500):
        x = _orbit(rng, rng.uniform(*e), 10.0 ** rng.uniform(np.log10(frac[0]), np.log10(frac[1])))
        assert lib.fixed_solve(T, *x, out.ctypes.data), x
        lib.errors(T, *x, out.ctypes.data, err.ctypes.data)
        worst = np.maximum(worst, np.abs(err))
    assert worst.max() <= 2.0 ** -53 * (1 + 2.0 ** -2), worst * 2.0 ** 53


def test_unbiased(lib):
    """f gdot - g fdot = 1: over many drifts the mean defect is far below one
    rounding (2^-60 per step would show after 1e9 steps)."""
    rng = np.random.default_rng(12)
    out = np.zeros(9)
    W = []
    for _ in range(20000):
        x = _orbit(rng, rng.uniform(0.0, 0.3), rng.uniform(0.02, 0.1))
        assert lib.fixed_solve(8, *x, out.ctypes.data)
        f1, g, fd, gd1 = (np.longdouble(v) for v in out[:4])
        W.append(float(g * fd - f1 - gd1 + f1 * gd1))
    W = np.asarray(W)
    assert abs(W.mean()) <= 4 * W.std() / np.sqrt(W.size) and W.std() < 2.0 ** -54


def test_left_to_the_general_solver(lib):
    """Unbound, near-parabolic, unresolved, degenerate and non-finite states."""
    out = np.zeros(9)
    ok = lambda *x: bool(lib.fixed_solve(8, *map(float, x), out.ctypes.data))
    h = 0.05 * 2 * np.pi
    assert ok(1, h, 1, 0, 1) and ok(1, h, 1, 0.1, 1)
    for x in [(1, h, 1, 0, 2), (1, h, 1, 0, 2.5), (1, h, 1, 0, 1.99999),          # escape speed and above
              (1, 2.0, 1, 0, 1), (1, h, 0.01, 0, 10), (1, h, 1, 4.0, 1.2),          # too long a step
              (1, h, 0, 0, 1), (1, h, np.inf, 0, 1), (1, h, np.nan, 0, 1), (1, h, 1, np.nan, 1),
              (1, h, 1, 0, np.nan), (1, h, 1, 0, np.inf), (1, h, 1e-320, 0, 1), (1, h, 1e200, 0, 1e-100),
              (1, 1e-300, 1, 0, 1), (1e-310, h, 1, 0, 1)]:
        assert not ok(*x), x
    # a parked lane: at rest, far away
    assert ok(1, 1e-3, 6.4e13, 0, 0) and out[0] > 0 and out[1] == 1e-3
    # scale invariance: lengths by 2^k, times by 2^l leave the coefficients' bits unchanged
    rng = np.random.default_rng(13)
    for _ in range(50):
        mu, h, r2, eta, v2 = _orbit(rng, 0.2, 0.05, a=1.0, mu=1.0)
        assert ok(mu, h, r2, eta, v2)
        ref = out.copy()
        k, l = int(rng.integers(-20, 20)), int(rng.integers(-20, 20))
        assert ok(np.ldexp(mu, 3 * k - 2 * l), np.ldexp(h, l), np.ldexp(r2, 2 * k), np.ldexp(eta, 2 * k - l),
                  np.ldexp(v2, 2 * k - 2 * l))
        assert out[0] == ref[0] and out[1] == np.ldexp(ref[1], l) and out[2] == np.ldexp(ref[2], -l) and out[3] == ref[3]
