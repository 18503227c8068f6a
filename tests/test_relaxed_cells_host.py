"""Cells that a step relaxes to their equilibrium from a small deviation (host build of
the integrator): the recombinations over the step against the ODE of the deviation,
integrated to 3e-14.

Tolerances.  FP64, 1e-12 relative: the closed form leaves out (b d)^3 / 300 of a term
that is d / 45 of the total (1e-13 at b d = 4e-3), and a few roundings add to it; slower
relaxation (q = 5) keeps the linearised form's (b d)^2 at b d = 1e-6.  Mixed: the same
at b d = 2e-2 is below a rounding; rounding of f at x0 and of the root leaves 1e-6."""
import itertools

import numpy as np
import pytest
from scipy.integrate import solve_ivp
from scipy.optimize import brentq

from test_integrator_host import SIG, lib  # noqa: F401  (the host build)

H = float(np.float32(3e9))


def _reference(A, b, c, x0):
    def F(x):
        return A * np.expm1(-b * x) + c * (1 - x) ** 2
    r = brentq(F, 0, 1, xtol=1e-300, rtol=4 * np.finfo(float).eps)
    o, e, d0 = 1 - r, A * np.exp(-b * r), x0 - r

    def f(t, s):
        d = s[0] * d0
        return [H * (e * np.expm1(-b * d) + c * (d * d - 2 * o * d)) / d0, H * c * (d * d - 2 * o * d)]
    return c * o * o * H + solve_ivp(f, (0, 1), [1.0, 0.0], method="DOP853", rtol=3e-14, atol=1e-20).y[1, -1]


@pytest.mark.parametrize("precision,tol,devs", [(0, 1e-12, [1e-6, 1e-4, 1e-3, 3.5e-3, -3.5e-3]),
                                                (1, 1e-6, [1e-3, 1e-2, 1.9e-2, -1.9e-2])])
def test_recombinations_of_relaxed_cells(lib, precision, tol, devs):  # noqa: F811
    n = 0
    for xe, b, q, y in itertools.product([0.05, 0.3, 0.9], [0.3, 1.0, 10.0], [46.0, 60.0, 300.0], devs):
        one = 1 - xe
        k = one * one / -np.expm1(-b * xe)
        c = q / (k * b * np.exp(-b * xe) + 2 * one) / H
        A, bb, x0 = k * c, b, xe + y / b
        if not 0 < x0 < 1:
            continue
        if precision:
            A, bb, c, x0 = (float(np.float32(v)) for v in (A, bb, c, x0))
        out = np.zeros(3)
        lib.oots_host_integrate_mono(precision, A, bb, 0.0, c, 0.0, SIG, x0, H, out.ctypes.data)
        ref = _reference(A, bb, c, x0)
        assert abs(out[1] / ref - 1) <= tol, (xe, b, q, y, out[1] / ref - 1)
        n += 1
    assert n > 60
