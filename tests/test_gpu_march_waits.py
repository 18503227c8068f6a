"""The march's bounded waits: a block that never publishes ends the call with an
error at every limit, however short, and the context works afterwards; no limit,
however large, ends a sound call."""
import numpy as np
import pytest

from paper_1201_5651_gb300 import inputs, oots

pytestmark = pytest.mark.gpu


def _context(scheme):
    w = inputs.small_random(n=70, ny=45, nz=50, seed=12, nsrc=1)
    w.sources[0].pos = (0.0, 0.0, 0.0)
    return w, oots.Context.from_workload(w, "mixed", scheme=scheme, K4=0.25)


@pytest.mark.parametrize("scheme", [oots.OOTS_A1, oots.OOTS_A3])
def test_waits_run_out_and_the_context_goes_on(scheme):
    w, c = _context(scheme)
    d = 1e-3 * w.t_rec
    c.step(d)
    want = c.get_neutral_fraction()
    for limit in (1, 3, 100):
        w, c = _context(scheme)
        c.debug_set(1, limit)
        c.debug_set(2, 0)
        with pytest.raises(oots.OotsError) as e:
            c.step(d)
        assert e.value.code == oots.OOTS_E_DEVICE_TIMEOUT
        c.debug_set(2, -1)
        c.debug_set(1, 1 << 22)
        c.reset_error()
        c.set_neutral_fraction(w.x0)
        c.set_time(0.0)
        c.step(d)
        assert np.array_equal(c.get_neutral_fraction(), want), limit


@pytest.mark.parametrize("limit", [1 << 59, 1 << 60, (1 << 63) - 1])
def test_large_limits_do_not_run_out(limit):
    w, c = _context(oots.OOTS_A3)
    c.debug_set(1, limit)
    c.step(1e-3 * w.t_rec)
