"""Cells over steps long against their recombination time, on the host build of the
integrator: near-neutral, weakly lit gas, whose recombination term grows from
nothing while its photoionisation changes little.  Against the ODE integrated to
3e-14 (Runge-Kutta of order 8): x(h), and with A1 the average attenuation.

Tolerances.  FP64: 1e-11, the host tests' bound.  Mixed: the quadrature stops at
1e-6 of the step, so x may be off by 1e-6 of its change, plus a few roundings of
6e-8: 1e-6; the average's logarithm carries b times that and its own rounding."""
import itertools

import numpy as np
import pytest
from scipy.integrate import solve_ivp

from test_integrator_host import SIG, lib  # noqa: F401  (the host build)

H = float(np.float32(3e9))


def _reference(A, b, c, x0):
    def f(t, y):
        x = x0 + y[0]
        return [H * (A * np.expm1(-b * x) + c * (1 - x) ** 2), np.expm1(-b * y[0])]
    y = solve_ivp(f, (0, 1), [0.0, 0.0], method="DOP853", rtol=3e-14, atol=1e-18).y[:, -1]
    return x0 + y[0], -b * x0 + np.log1p(y[1])


@pytest.mark.parametrize("x0", [1 - 1e-6, 0.999, 0.99, 0.9])
def test_near_neutral_cells_over_long_steps(lib, x0):  # noqa: F811
    for ch, b, g in itertools.product([0.1, 0.3, 1, 3, 10, 30], [0.01, 0.1, 0.3, 1, 3], [0.01, 0.07, 0.15]):
        A, bb, c, x = (float(np.float32(v)) for v in (g / b / H, b, ch / H, x0))
        xr, lr = _reference(A, bb, c, x)
        for b0 in (0.0, bb):
            for precision, tol in ((0, 1e-11), (1, 1e-6)):
                out = np.zeros(3)
                lib.oots_host_integrate_mono(precision, A, bb, 0.0, c, b0, SIG, x, H, out.ctypes.data)
                assert abs(out[0] - xr) <= tol, (precision, x0, ch, b, g, b0, out[0] - xr)
                if b0 > 0:
                    assert abs(out[2] - lr) <= tol * max(1.0, bb), (precision, x0, ch, b, g, out[2] - lr)
