"""The interaction sub-step: its float-pair arithmetic (csrc/whg_interact.cuh) on
the CPU against 113-bit arithmetic, and on the GPU the systems at the edges
of that form against the oracle."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2307_05683_gb300 import inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#include "whg_interact.cuh"
#if defined(__aarch64__)
typedef long double Q;
#else
typedef __float128 Q;
#endif
using namespace whg;
static Q root(Q x) { Q y = sqrt((double)x); for (int i = 0; i < 4; ++i) y = (y + x / y) / 2; return y; }
static long long grid(double q, int e)
{
    const fixed::u64 b = fixed::bits_of(q);
    return fixed::to_fixed(b, 5 + e - fixed::exponent_of(b));
}
// Relative errors of the kick of a mass factor hm over the separation b - a
// (power 3) or of the GR kick at a (power 4), positions taken on their grid.
extern "C" double kick_error(int power, double hm, const double* a, const double* b)
{
    int e = 0;
    for (int c = 0; c < 3; ++c) {
        e = fixed::exponent_of(fixed::bits_of(a[c])) > e ? fixed::exponent_of(fixed::bits_of(a[c])) : e;
        e = fixed::exponent_of(fixed::bits_of(b[c])) > e ? fixed::exponent_of(fixed::bits_of(b[c])) : e;
    }
    long long A[3], B[3];
    pairs::Coord ca[3], cb[3];
    for (int c = 0; c < 3; ++c) {
        A[c] = grid(a[c], e);
        B[c] = grid(b[c], e);
        ca[c] = pairs::chunks(A[c]);
        cb[c] = pairs::chunks(B[c]);
    }
    pairs::Pair d[3];
    Q x[3], r2 = 0;
    for (int c = 0; c < 3; ++c) {
        d[c] = power == 3 ? pairs::difference(cb[c], ca[c]) : pairs::own(ca[c]);
        x[c] = (Q)(power == 3 ? B[c] - A[c] : A[c]) / ((Q)(1 << 20) * (1 << 20));
        r2 += x[c] * x[c];
    }
    const pairs::Separation s = pairs::separation(d[0], d[1], d[2]);
    if (power == 4) hm = ldexp(hm, 1040 - e);            // as the kernel scales the GR factor
    const pairs::Pair w = pairs::product(pairs::split(hm), power == 3 ? pairs::inverse_cube(s) : pairs::inverse_fourth(s));
    const Q p = power == 3 ? r2 * root(r2) : r2 * r2;
    double off = 0, all = 0;
    for (int c = 0; c < 3; ++c) {
        const pairs::Pair f = pairs::product(w, d[c]);
        const Q exact = (Q)hm * x[c] / p, err = (Q)f.h + f.l - exact;
        off += (double)(err * err);
        all += (double)(exact * exact);
    }
    return sqrt(off / all);
}
extern "C" double widened(float f, int k) { return pairs::widen(f, k); }
extern "C" double summed(const float* f, int n)
{
    pairs::Pair s = {0.0f, 0.0f};
    for (int i = 0; i < n; ++i) pairs::accumulate(s, f[2 * i], f[2 * i + 1]);
    return (double)s.h + (double)s.l;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("pairs")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-O1", "-std=gnu++17", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2307_05683_gb300", "csrc"), str(src), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    lib.kick_error.restype = lib.widened.restype = lib.summed.restype = ctypes.c_double
    lib.kick_error.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_void_p, ctypes.c_void_p]
    lib.widened.argtypes = [ctypes.c_float, ctypes.c_int]
    lib.summed.argtypes = [ctypes.c_void_p, ctypes.c_int]
    return lib


@pytest.mark.parametrize("power", [3, 4])
@pytest.mark.parametrize("sep", [1.0, 1e-2, 1e-4])
def test_kick_terms_against_113_bits(lib, power, sep):
    """A term's error is a few roundings of 2^-46 (the low parts' last bits):
    at most 2^-42, and 2^-45 in the mean square; a separation of 1e-4 of the
    grid has 6 bits fewer in its worst coordinate, 2^-36."""
    rng = np.random.default_rng(3)
    err = []
    for _ in range(3000):
        size = 10.0 ** rng.uniform(-2, 2)
        a = rng.uniform(-1, 1, 3) * size
        b = a + rng.uniform(-1, 1, 3) * size * sep
        err.append(lib.kick_error(power, 10.0 ** rng.uniform(-12, -3), a.ctypes.data, b.ctypes.data))
    err = np.asarray(err)
    tight = sep >= 1e-2 or power == 4
    assert err.max() <= 2.0 ** (-42 if tight else -36), np.log2(err.max())
    assert np.sqrt((err ** 2).mean()) <= 2.0 ** (-45 if tight else -42)


def test_sums_and_conversion(lib):
    rng = np.random.default_rng(4)
    for _ in range(200):
        n = int(rng.integers(1, 8))
        h = (rng.normal(size=n) * 10.0 ** rng.uniform(-6, 6, n)).astype(np.float32)
        f = np.stack([h, (h * rng.uniform(-1, 1, n) * 2.0 ** -24).astype(np.float32)], 1)
        exact = f.astype(np.float64).sum(axis=0, dtype=np.longdouble).sum()
        got = lib.summed(np.ascontiguousarray(f).ctypes.data, n)
        assert abs(got - float(exact)) <= 2.0 ** -44 * np.abs(h.astype(np.float64)).max()
    for x in [0.0, 1.0, -1.0, 3.1415927, -2.0 ** -100, 1.9999999 * 2.0 ** 30]:
        for k in (-60, -1, 0, 1, 60):
            x32 = float(np.float32(x))
            assert lib.widened(x32, k) == np.ldexp(x32, k)
    assert lib.widened(1e-40, 0) == 0.0                  # FP32 subnormals count as 0


# ------------------------------------------------------------------- GPU --

def _system(kind, n, seed, S=24):
    """Star + n planets, every system drawn anew."""
    rng = np.random.default_rng(seed)
    a = 0.5 * 1.6 ** np.arange(n) * np.ones((S, 1))
    m = 10.0 ** rng.uniform(-6, -4, (S, n))
    M = rng.uniform(0, 2 * np.pi, (S, n))
    frac = 1.0 / 25.0
    if kind == "heavy":                                  # a companion of the star's order
        a = a * np.where(np.arange(n) == n - 1, 6.0, 1.0)
        m[:, -1] = 0.3
    elif kind == "strong":                               # kicks around the accepted 2^-11 of the velocity
        m = 10.0 ** rng.uniform(-3.5, -2.5, (S, n))
    elif kind == "near":                                 # two planets 1e-3 apart, almost massless
        m = m * 1e-7
        a[:, 1] = a[:, 0] * 1.001
        M[:, 1] = M[:, 0] + 1e-3
    elif kind == "wide":                                 # 0.02 to 2000
        a = 0.02 * (2000 / 0.02) ** (np.arange(n) / max(1, n - 1)) * np.ones((S, 1))
    elif kind == "massless":
        m[:, ::2] = 0.0
    elif kind == "small":                                # lengths below the grid's range: all in FP64
        a = a * 1e-7
    e, inc = rng.uniform(0, 0.05, (S, n)), rng.uniform(0, 0.05, (S, n))
    ang = rng.uniform(0, 2 * np.pi, (2, S, n))
    x, v = inputs.elements_to_state(1.0 + m, a, e, inc, ang[0], ang[1], M)
    if kind == "near":                                   # the same node and pericentre
        x[:, 1], v[:, 1] = inputs.elements_to_state(1.0, a[:, 1], e[:, 0], inc[:, 0], ang[0][:, 0], ang[1][:, 0],
                                                    M[:, 1])
    dt = 2 * np.pi * np.sqrt(a[:, 0] ** 3) * frac
    return inputs._assemble(1.0, m, x, v, np.full(S, n), dt, kind)


@pytest.mark.gpu
@pytest.mark.parametrize("gr", [0, 1, 2])
@pytest.mark.parametrize("n", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("kind", ["plain", "heavy", "strong", "near", "wide", "massless", "small"])
def test_sub_step_edges_match_oracle(orc, kind, n, gr):
    """One and 30 steps against the oracle, 1e-12 and 1e-11 of each system's
    largest coordinate, for systems inside the float-pair form, outside it and
    on its edge, every lane-group size, lanes without a planet among them."""
    from paper_2307_05683_gb300 import build, whg
    build.build()
    ens = _system(kind, n, 100 * n + gr)
    # a light speed of 100 orbital velocities at the innermost planet: GR counts
    c = 100.0 / np.sqrt(_inner(kind))
    for steps, tol in ((1, 1e-12), (30, 1e-11)):
        it = whg.Integrator(ens.n_systems, n, gr_mode=gr, c_light=c)
        it.init(ens)
        it.step(steps)
        p, v, st, t = it.read_state()
        it.close()
        o = orc.OracleEnsemble(ens.n_systems, n, gr_mode=gr, c_light=c)
        o.init(ens)
        o.step(steps)
        po, vo, so, to = o.read_state()
        assert np.array_equal(st, so) and np.allclose(t, to, rtol=1e-15, atol=0)
        scale = np.abs(po).max(axis=(1, 2))[:, None, None]
        assert (np.abs(p - po) / scale).max() <= tol
        scale = np.abs(vo).max(axis=(1, 2))[:, None, None]
        assert (np.abs(v - vo) / scale).max() <= tol


def _inner(kind):
    return {"wide": 0.02, "small": 0.5e-7}.get(kind, 0.5)
