"""Steps of one and of several recombination times in near-neutral gas, each scheme
against the oracle: A1 under its own criterion K1 = 1 (a step of exactly one
recombination time), A2 and A3 over five."""
import numpy as np
import pytest

import oracle
from paper_1201_5651_gb300 import inputs, oots

pytestmark = pytest.mark.gpu

# FP64: the bound of every FP64 step.  Mixed: columns agree to 1e-5 and enter the state with a factor below
# two (optical depths of a few).
TOL = {"fp64": 1e-9, "mixed": 2e-5}


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("scheme,steps", [(oots.OOTS_A1, 1.0), (oots.OOTS_A2, 5.0), (oots.OOTS_A3, 5.0)])
def test_long_step_matches_oracle(precision, scheme, steps):
    # cells of optical depth 0.2 and light so weak that it moves most of them by a few per cent a step
    w = inputs.small_random(n=22, ny=20, nz=18, seed=6, nsrc=1, Q=5e37, box_rs=4.2)
    w.nH = np.full_like(w.nH, 100.0)
    w.uniform_n = 100.0
    w.x0 = np.full_like(w.x0, 1 - 1e-6)
    d = steps * w.t_rec
    c = oots.Context.from_workload(w, precision, scheme=scheme, **({"K1": 1.0} if scheme == oots.OOTS_A1 else {"K4": 0.25}))
    if scheme == oots.OOTS_A1:
        assert abs(c.compute_dt() / w.t_rec - 1) <= 1e-5
    c.step(d)
    x = np.ascontiguousarray(w.x0.astype(np.float64))
    oracle.Problem.from_workload(w).substep(x, 0.0, d, scheme=scheme, dt_fixed=d)
    got = c.get_neutral_fraction()
    assert np.mean((x > 0.9) & (x < 0.999)) > 0.3
    assert float(np.max(np.abs(got - x))) <= TOL[precision]
