"""A batched FP32 cell's averages are FP64 sums of its field values.

Elastic cells whose phases differ by 1e5 in stiffness: the stresses of one
cell span more than 2^16, so a sum carried in a pair of FP32 values (about
2^-48 of it) loses bits that FP64 keeps.  On such values, in the chunk order
of the kernels, the rounding of FP64 sums is 2e-17 of the mean magnitude (rms,
emulated in numpy) and that of FP32 pairs 2e-15; the bound lies a factor of
ten above the former.  512 voxels: the division by their number is exact.
"""
import math

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _cell(seed):
    rng = np.random.default_rng(seed)
    n = (8, 8, 8)
    rows = [dict(W.generators._matrix_row(k), elastic=1) for k in (1.0, 1e5)]
    phase = (rng.uniform(size=n) < 0.5).astype(np.uint16)
    E, G = 0.004 * rng.standard_normal((3, 3)), 0.002 * rng.standard_normal((3, 3))
    time, Ep, Gp = W.ramp_path(1, E, G)
    return W.generators._problem(n, phase, W.phase_record(rows), time, Ep, Gp, 1e-6, ref_kind="midrange")


def test_averages_are_fp64_sums():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2409_10774_gb300 as M
    cells = [_cell(s) for s in range(6)]
    off = []
    for r in M.mp_batch_solve(M.Context(0), cells, precision=1, fields=True, lockstep_iters=[[3]] * len(cells)):
        assert r["status"] == "ok"
        for mean, field in (("T", "t"), ("M", "m"), ("Eavg", "e"), ("Gavg", "g")):
            values = r["final"][field].reshape(512, 9)
            for c in range(9):
                exact = math.fsum(values[:, c]) / 512.0
                off.append((r[mean][-1].reshape(9)[c] - exact) / np.abs(values[:, c]).mean())
    assert np.sqrt(np.mean(np.square(off))) <= 2e-16
