"""The column march at the edges of its blocks (32 lanes, 7 or 21 rows, chunks of
eight layers): sides one short of, equal to and one past those sizes, sources on
corners, faces and inside, with one array (uniform density), two (density and
state) and packed input (four sources and more, rows padded to eight)."""
import numpy as np
import pytest

import oracle
from paper_1201_5651_gb300 import inputs, oots

pytestmark = pytest.mark.gpu


def _rel(a, b, floor=1e10):
    return float(np.max(np.abs(a - b) / np.maximum(np.abs(b), floor)))


# FP64: a column is a sum of at most ~130 positive increments, interpolated with weights that sum to one:
# a few hundred roundings of 1e-16.  Mixed: increments, weights and the result are floats (6e-8 each), and
# a weighted difference of neighbouring columns loses up to two digits more beside a vertex.
TOL = {"fp64": 1e-12, "mixed": 1e-5}


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dims,pos", [
    ((1, 1, 1), (0, 0, 0)), ((9, 1, 1), (4, 0, 1)), ((33, 8, 7), (0, 0, 0)), ((32, 32, 32), (0, 0, 0)),
    ((65, 22, 43), (65, 0, 21)), ((8, 66, 21), (3, 33, 0)), ((20, 15, 70), (13, 7, 37)), ((64, 63, 31), (31, 32, 16)),
])
def test_columns_at_block_edges(precision, dims, pos):
    w = inputs.small_random(n=dims[0], ny=dims[1], nz=dims[2], seed=31 + sum(dims), nsrc=1)
    w.sources[0].pos = tuple(float(p) for p in pos)
    for uniform in (False, True):
        if uniform:
            w.nH = np.full_like(w.nH, 100.0)
            w.uniform_n = 100.0
        c = oots.Context.from_workload(w, precision, scheme=oots.OOTS_A3, K4=0.25)
        c.compute_dt()
        assert _rel(c.get_column_density(0), oracle.Problem.from_workload(w).trace(0, w.x0)) <= TOL[precision], uniform


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nx,nsrc", [(37, 4), (40, 5), (7, 9)])
def test_packed_columns_and_repeated_traces(precision, nx, nsrc):
    """Packed rows, and a second and third trace of the same launch set bit for bit as the first."""
    w = inputs.small_random(n=nx, ny=34, nz=23, seed=5 + nx, nsrc=nsrc)
    c = oots.Context.from_workload(w, precision, scheme=oots.OOTS_A3, K4=0.25)
    P = oracle.Problem.from_workload(w)
    first = None
    for _ in range(3):
        c.compute_dt()
        got = [c.get_column_density(s) for s in range(nsrc)]
        if first is None:
            first = got
            for s in range(nsrc):
                assert _rel(got[s], P.trace(s, w.x0)) <= TOL[precision], s
        else:
            assert all(np.array_equal(a, b) for a, b in zip(first, got))


@pytest.mark.parametrize("dims,pos,spectrum", [
    ((33, 9, 15), (0, 0, 0), "mono"), ((7, 34, 8), (3, 34, 4), "bb"), ((14, 15, 32), (14, 0, 16), "mono"), ((1, 9, 1), (0, 4, 0), "bb"),
])
def test_a1_at_block_edges_fp64(dims, pos, spectrum):
    """A1 (blocks of 32 x 7 cells, a hand-off per layer): state and entry columns after one step against the
    oracle.  1e-9 as every FP64 step: cells integrate to 1e-13 there and here, columns sum ~40 of them."""
    w = inputs.small_random(n=dims[0], ny=dims[1], nz=dims[2], seed=3 + sum(dims), nsrc=1, spectrum=spectrum)
    w.sources[0].pos = tuple(float(p) for p in pos)
    d = 0.05 * w.t_rec
    c = oots.Context.from_workload(w, "fp64", scheme=oots.OOTS_A1, dt_fixed=d)
    c.step(d)
    x = np.ascontiguousarray(w.x0.astype(np.float64))
    _, _, bud, _ = oracle.Problem.from_workload(w).substep(x, 0.0, d, scheme=1, dt_fixed=d)
    assert float(np.max(np.abs(c.get_neutral_fraction() - x))) <= 1e-9
    assert np.allclose(c.get_budget(), bud, rtol=1e-8)      # tied cells are counted once


@pytest.mark.parametrize("ny,nz", [(22, 23), (24, 22), (60, 66), (72, 65)])
def test_a1_plane_rows_on_both_sides_of_the_group_rule(ny, nz):
    """506 rows take a lane group each, 528 and more a thread each: all follow the oracle (1e-9, as above)."""
    w = inputs.plane_random(n=6, ny=ny, nz=nz, seed=8, axis=0, x_lo=0.2)
    d = 0.02 * w.t_rec
    c = oots.Context.from_workload(w, "fp64", scheme=oots.OOTS_A1, dt_fixed=d)
    c.step(d)
    x = np.ascontiguousarray(w.x0.astype(np.float64))
    oracle.Problem.from_workload(w).substep(x, 0.0, d, scheme=1, dt_fixed=d)
    assert float(np.max(np.abs(c.get_neutral_fraction() - x))) <= 1e-9
