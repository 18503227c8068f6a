"""A context of a batch that is asked for its time while the batch's substeps are
still running: the answer may be of any moment, but nothing that follows goes by
it.  The run that was asked ends where the run that was not asked ends."""
import numpy as np
import pytest

from paper_1201_5651_gb300 import inputs, oots

pytestmark = pytest.mark.gpu


def _batch():
    ws = [inputs.small_random(n=n, seed=n, nsrc=1) for n in (40, 36, 33)]
    ctxs = [oots.Context.from_workload(w, "mixed", scheme=oots.OOTS_A3, K4=0.25) for w in ws]
    return ws, ctxs, oots.Batch(ctxs)


def _end(ask):
    ws, ctxs, b = _batch()
    b.run_substeps(200, [1e30] * 3)
    if ask:
        for c in (ctxs[1], ctxs[2]):
            c.get_time()
            c.get_budget()
    ctxs[0].synchronize()
    b.close()
    ctxs[1].step(1e-3 * ws[1].t_rec)
    ctxs[2].compute_dt()
    return [(c.get_time(), c.get_budget(), c.get_neutral_fraction()) for c in ctxs]


def test_early_question_leaves_the_state_alone():
    for (t, bud, x), (t1, bud1, x1) in zip(_end(False), _end(True)):
        assert t == t1
        assert np.allclose(bud, bud1, rtol=1e-9)
        assert np.array_equal(x, x1)


def test_substeps_counted_after_an_early_question():
    t = [c[0][0] for c in _end(False)]
    _, ctxs, b = _batch()
    b.run_substeps(200, [1e30] * 3)
    for c in reversed(ctxs):                     # the first context, on whose stream the batch runs, last
        c.get_time()
    n = b.advance([1.2 * v for v in t])
    assert [c.get_time()[1] for c in ctxs] == [200 + m for m in n]
    b.close()
