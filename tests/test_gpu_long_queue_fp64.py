"""FP64 grids whose queue of the general pass is longer than its thread-per-cell rule
(40960 cells), with one source and with several, against the oracle on a sample:
1e-10, the host tests' bound for random cells of the same integrator."""
import numpy as np
import pytest

import oracle
from paper_1201_5651_gb300 import inputs, oots

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [33, 38])             # 36 k cells: lane groups; 55 k, nearly all queued: threads
@pytest.mark.parametrize("nsrc", [1, 3])
def test_queue_on_both_sides_of_the_rule(n, nsrc):
    w = inputs.small_random(n=n, ny=n, nz=n, seed=3, nsrc=nsrc, spectrum="bb", Q=1e52, x_lo=0.02, box_rs=0.02)
    d = 0.002 * w.t_rec
    c = oots.Context.from_workload(w, "fp64", scheme=oots.OOTS_A2, dt_fixed=d)
    c.step(d)
    x = c.get_neutral_fraction().ravel()
    N = np.stack([c.get_column_density(s) for s in range(nsrc)])
    idx = np.random.default_rng(1).choice(w.ncell, 200, replace=False)
    ref = oracle.Problem.from_workload(w).integrate_cells(idx, w.x0.ravel()[idx], N, d)
    assert float(np.max(np.abs(x[idx] - ref))) <= 1e-10
