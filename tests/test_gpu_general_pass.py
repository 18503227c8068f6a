"""The general integration pass on both sides of its thread-per-cell rule (65536
queued cells of a grid), alone and in a batch that mixes both kinds of grid, and
the series step of slow cells against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1201_5651_gb300 import inputs, oots

pytestmark = pytest.mark.gpu


def _workload(n, seed, nsrc):
    """Random states and a strong source: most cells need the general pass."""
    return inputs.small_random(n=n, ny=n, nz=n, seed=seed, nsrc=nsrc, Q=1e52, x_lo=0.02, box_rs=0.02)


@pytest.mark.parametrize("nsrc", [1, 3])
def test_long_queue_alone_and_in_a_mixed_batch(nsrc):
    """One grid whose queue is long and one whose queue is short: each ends where its own run ends, bit for
    bit.  The long one is checked cell by cell against the oracle on a sample: the mixed path integrates to
    float rounding, and 1e-4 is the bound of the host tests of the same integrator."""
    ws = [_workload(60, 3, nsrc), _workload(12, 4, nsrc)]
    dt = [0.002 * w.t_rec for w in ws]
    solo = []
    for w, d in zip(ws, dt):
        c = oots.Context.from_workload(w, "mixed", scheme=oots.OOTS_A2, dt_fixed=d)
        c.advance(d)
        solo.append((c.get_neutral_fraction(), c.get_budget(),
                     np.stack([c.get_column_density(s) for s in range(nsrc)])))
    ctxs = [oots.Context.from_workload(w, "mixed", scheme=oots.OOTS_A2, dt_fixed=d) for w, d in zip(ws, dt)]
    b = oots.Batch(ctxs)
    b.advance(dt)
    b.close()
    for c, (x, bud, _) in zip(ctxs, solo):
        assert np.array_equal(c.get_neutral_fraction(), x)
        assert np.allclose(c.get_budget(), bud, rtol=1e-5)
    w, (x, _, N) = ws[0], solo[0]
    idx = np.random.default_rng(1).choice(w.ncell, 400, replace=False)
    P = oracle.Problem.from_workload(w)
    ref = P.integrate_cells(idx, w.x0.ravel()[idx], N, dt[0])
    assert float(np.max(np.abs(x.ravel()[idx] - ref))) <= 1e-4


@pytest.mark.parametrize("spectrum", ["mono", "bb"])
@pytest.mark.parametrize("scale", [1e-5, 1e-3, 3e-2])
def test_slow_cells_fp64(spectrum, scale):
    """Steps so short that cells pass from the linearised step to the series to the quadrature: 1e-11 per
    cell in FP64 (the oracle integrates to 1e-13, columns agree to 1e-12)."""
    w = inputs.small_random(n=22, ny=21, nz=20, seed=9, nsrc=1, spectrum=spectrum, x_lo=0.3)
    c = oots.Context.from_workload(w, "fp64", scheme=oots.OOTS_A2, K4=0.25)
    d = scale * c.compute_dt()
    c.step(d)
    x = np.ascontiguousarray(w.x0.astype(np.float64))
    oracle.Problem.from_workload(w).substep(x, 0.0, d, scheme=2, dt_fixed=d)
    assert float(np.max(np.abs(c.get_neutral_fraction() - x))) <= 1e-11
