"""Closed-form passes over runs of cells: a block's run holds 1 to 16 times its
threads by the size of the call, starts anywhere in a grid and may hold several
grids.  A cell's arithmetic does not depend on where its run begins, so a grid
gives the same bits alone (short runs) and in a batch large enough for long
runs; the budgets are sums in another order."""
import numpy as np
import pytest

from paper_1201_5651_gb300 import inputs, oots

pytestmark = pytest.mark.gpu


def _contexts(precision, nsrc, spectrum):
    sizes = [(7, 7, 7), (33, 5, 3), (1, 1, 130), (129, 1, 1), (64, 32, 8), (190, 173, 160)]
    ws = [inputs.small_random(n=nx, ny=ny, nz=nz, seed=5 + nx, nsrc=nsrc, spectrum=spectrum) for nx, ny, nz in sizes]
    return ws, [oots.Context.from_workload(w, precision, scheme=3, K4=0.25) for w in ws]


@pytest.mark.parametrize("precision,nsrc,spectrum", [("mixed", 1, "mono"), ("mixed", 1, "bb"), ("mixed", 3, "bb"),
                                                      ("fp64", 1, "mono")])
def test_runs_match_solo(precision, nsrc, spectrum):
    ws, solo = _contexts(precision, nsrc, spectrum)
    for c in solo:
        c.run_substeps(2, 1e30)
    _, batched = _contexts(precision, nsrc, spectrum)
    b = oots.Batch(batched)
    b.run_substeps(2, [1e30] * len(batched))
    for i, (c, d) in enumerate(zip(solo, batched)):
        assert np.array_equal(c.get_neutral_fraction(), d.get_neutral_fraction()), i
        assert c.get_time() == d.get_time(), i
    b.close()
