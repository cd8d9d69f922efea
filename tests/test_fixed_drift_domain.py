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
