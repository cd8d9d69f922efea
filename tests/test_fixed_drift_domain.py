"""The edges of the fixed-point Kepler solver's domain (csrc/whg_fixed.cuh), on
the CPU."""
import numpy as np
import pytest

from test_fixed_drift import lib  # noqa: F401  (fixture: the solver's host build)


@pytest.mark.parametrize("log2v", [11, 63, 64, 65, 70, 80, 91, 100, 128, 160, 192, 200, 256, 299])
@pytest.mark.parametrize("cosine", [0.0, 1e-30, 0.3, -0.7, 1.0])
def test_unbound_speeds_of_any_size_are_left_out(lib, log2v, cosine):  # noqa: F811
    """v^2 h^2/r0^2 from 2^14 to far beyond FP32's range: an orbit that is not
    bound, whichever way it moves."""
    out = np.zeros(9)
    v = 2.0 ** log2v
    assert not lib.fixed_solve(8, 1.0, 0.05, 1.0, cosine * v, v * v, out.ctypes.data)


@pytest.mark.parametrize("log2r,log2h,log2mu", [(-40, 40, 0), (-90, 60, 0), (-60, 60, 90), (-99, 149, 99), (-99, 10, -99)])
def test_unresolved_steps_of_any_size_are_left_out(lib, log2r, log2h, log2mu):  # noqa: F811
    """mu h^2/r0^3 from 2^200 to 2^694."""
    out = np.zeros(9)
    r, h, mu = 2.0 ** log2r, 2.0 ** log2h, 2.0 ** log2mu
    for v2 in (0.0, 0.25 * mu / r, mu / r):
        assert not lib.fixed_solve(8, mu, h, r * r, 0.0, v2, out.ctypes.data)


@pytest.mark.parametrize("T", [6, 8])
@pytest.mark.parametrize("zmin", [0.0, 0.5, 1.0, 1.5])
def test_coefficients_over_the_whole_domain(lib, T, zmin):  # noqa: F811
    """m, V and a drawn over all that the solver takes (z from zmin to zmin +
    0.5).  1 - f, fdot and 1 - gdot are one rounding (2^-53 of the value at
    most, 0.43 2^-53 rms and no mean) away from a value of 55 correct bits, and
    unbiased: mean within 2^-57 and the sample's own scatter.  g is h times a
    difference from 1 of such a value, so it is judged against h."""
    rng = np.random.default_rng(21)
    out, err, kept = np.zeros(9), np.zeros(9), []
    while len(kept) < 3000:
        m = rng.uniform(0, 4)
        V, a = 2 * m * rng.uniform(), rng.uniform(-1, 1)
        r0 = rng.uniform(1, 2)
        h = np.sqrt(m * r0 ** 3)
        x = (1.0, h, r0 * r0, a * r0 * r0 / h, V * r0 * r0 / (h * h))
        if a * a > V or not lib.fixed_solve(T, *x, out.ctypes.data):
            continue
        z = (2 * m - V) * out[4] ** 2
        if zmin <= z < zmin + 0.5:
            lib.errors(T, *x, out.ctypes.data, err.ctypes.data)
            kept.append([err[0], err[1] * out[1] / h, err[2], err[3]])
    e = np.asarray(kept) * 2.0 ** 53
    assert np.abs(e).max() <= 1.25, np.abs(e).max(axis=0)
    assert np.sqrt((e ** 2).mean(axis=0)).max() <= 0.5
    assert np.all(np.abs(e.mean(axis=0)) <= 2.0 ** -4 + 4 * e.std(axis=0) / np.sqrt(len(e))), e.mean(axis=0)
