"""Tiles of several columns and items of several rows, cut off at the end.

A cell on its own mostly gets y / z tiles of one column, batched cells full
tiles (256 / n columns of length n in FP32, 128 / n in FP64, at least one), so
a batch of thin boxes takes the line kernels through several columns, the gap
between their stages, short last tiles, three-stage plans and flat cells (all
18 fields through z), each beside cells of other lengths.  Single cells with
more (y, z) rows than SMs take pass A's items through several rows with a last
item cut off.  One plastic increment with a prescribed number of iterations,
against the FP64 oracle; tolerances as in test_gpu_parity_lengths.py.
"""
import numpy as np
import pytest

import workloads as W
from parity_helpers import compare_solves
from oracle import solver as OS

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ITERATIONS = 5
_REFERENCE = {}


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2409_10774_gb300 as M
    c = M.Context(0)
    c.set_autotune(False)  # the default rows per item
    return c


def _problem(n):
    rng = np.random.default_rng([7, *n])
    phase = (rng.uniform(size=(n[2], n[1], n[0])) < 0.35).astype(np.uint16)
    rows = [dict(W.generators._matrix_row()), dict(W.generators._matrix_row(2.0), elastic=1)]
    time, E, G = W.ramp_path(1, np.array([[0.004, 0.001, 0.0], [0.0, -0.001, 0.0], [0.0, 0.0, 0.001]]),
                             np.array([[0.0, 0.001, 0.0], [0.0, 0.0, 0.0], [0.0, 0.0, 0.002]]))
    return W.generators._problem(n, phase, W.phase_record(rows), time, E, G, 1e-9, ref_kind="midrange")


def _reference(n):
    if n not in _REFERENCE:
        _REFERENCE[n] = OS.solve(_problem(n), lockstep_iters=[ITERATIONS])
        assert _REFERENCE[n]["status"] == "ok" and _REFERENCE[n]["P"][0] > 0.0
    return _REFERENCE[n]


def _compare(res, n, precision):
    assert res["status"] == "ok"
    compare_solves(res, _reference(n), *((1e-11, 1e-11) if precision == 0 else (1e-6, 1e-5)))


def _tiles(n, precision):
    """(columns, columns per full tile) of the y and z passes of a batched cell."""
    kx = max(1, n[0] // 2)
    full = [max(1, (256 if precision else 128) // length) for length in n[1:]]
    return (n[2] * kx, full[0]), (n[1] * kx, full[1])


# axis under test: 0 = y, 1 = z; whether FP32 / FP64 tiles hold several columns
# and whether the last one is cut off
CUT, FULL, ONE = "cut", "full", "one"
BATCH = [
    ((2, 36, 8), 0, CUT, CUT), ((2, 8, 36), 1, CUT, CUT),
    ((18, 54, 1), 0, CUT, CUT), ((6, 6, 54), 1, CUT, FULL),
    ((2, 72, 4), 0, CUT, ONE), ((2, 4, 72), 1, CUT, ONE),
    ((18, 96, 1), 0, CUT, ONE), ((6, 4, 96), 1, FULL, ONE),
    ((18, 108, 1), 0, CUT, ONE), ((6, 4, 108), 1, FULL, ONE),
    ((6, 12, 18), 1, CUT, CUT), ((6, 18, 24), 0, CUT, CUT), ((6, 6, 24), 1, CUT, CUT),
    # flat cells: the z pass on 18 fields
    ((18, 1, 54), 1, CUT, CUT), ((18, 1, 96), 1, CUT, ONE), ((18, 1, 48), 1, CUT, CUT),
    # three stages; 384 is the longest FP64 column
    ((2, 384, 4), 0, ONE, ONE), ((2, 4, 384), 1, ONE, ONE),
]


def test_batch_cases_have_the_tiles_they_claim():
    for n, axis, fp32, fp64 in BATCH:
        for precision, claim in ((1, fp32), (0, fp64)):
            columns, full = _tiles(n, precision)[axis]
            kind = ONE if full == 1 else CUT if columns % full and columns > full else FULL
            assert columns >= full or kind == ONE
            assert kind == claim, (n, precision, columns, full)


@pytest.mark.parametrize("precision", [0, 1])
def test_batched_boxes(ctx, precision):
    import paper_2409_10774_gb300 as M
    sizes = [case[0] for case in BATCH] + ([(2, 432, 4), (2, 4, 486), (2, 512, 2), (2, 2, 512)] if precision else [])
    res = M.mp_batch_solve(ctx, [_problem(n) for n in sizes], precision=precision, fields=True,
                           lockstep_iters=[[ITERATIONS]] * len(sizes))
    for n, r in zip(sizes, res):
        _compare(r, n, precision)


# (grid, rows per item FP32 / FP64): 1 where a row fills an item
@pytest.mark.parametrize("n, rows", [((6, 4, 8), (6, 6)), ((18, 12, 54), (5, 5)), ((36, 12, 54), (5, 3)),
                                     ((36, 16, 32), (4, 3)), ((54, 1, 486), (4, None)), ((72, 16, 32), (3, 1)),
                                     ((48, 12, 54), (5, 2)), ((96, 12, 16), (2, 1)), ((108, 12, 16), (2, 1))])
@pytest.mark.parametrize("precision", [0, 1])
def test_rows_per_item(ctx, n, rows, precision):
    import paper_2409_10774_gb300 as M
    want = rows[1 - precision]
    if want is None:
        pytest.skip("an FP64 column of 486 points does not fit a tile")
    rve = M.Rve(ctx, _problem(n), precision=precision, lockstep_iters=[ITERATIONS])
    assert rve.config()["rows_per_item"] == want
    assert rve.run(1) == 0
    res = rve.results(fields=True)
    rve.close()
    _compare(dict(res, status="ok"), n, precision)
