"""The y and z passes on every supported axis length (each has its own
compile-time plan), against the FP64 oracle.

A length L is put on y and on z of a thin cell, next to an axis of another
length, so that tiles hold one column or several, full and cut off, and the
reduced fields of the z pass meet every plan; N2 = 1 takes the z pass on all
18 fields.  Tolerances as in test_gpu_parity.py: 1e-12 (FP64) and 2e-6 (FP32)
per unit of rounding growth, times 10.
"""
import numpy as np
import pytest

from oracle import constitutive as OC
from oracle import fft as OF
from oracle.green import GreenOperator, wavevectors

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LENGTHS = (2, 4, 6, 8, 12, 16, 18, 24, 32, 36, 48, 54, 64, 72, 96, 108, 128, 144, 162, 192, 216, 256, 288, 324,
           384, 432, 486, 512)


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2409_10774_gb300 as M
    return M.Context(0)


def _check(ctx, n, precision):
    import paper_2409_10774_gb300 as M
    rng = np.random.default_rng(sum(n) * 17 + precision)
    shape = (n[2], n[1], n[0], 3, 3)
    tau, mu = rng.standard_normal(shape), rng.standard_normal(shape)
    h, ref = 0.83, (20.0, 12.0, 3.0, 0.7, 1.1, 1.9)
    xi, active = wavevectors(n, h)
    op = GreenOperator(xi, active, OC.stiffness_A(*ref[:3]), OC.stiffness_B(*ref[3:]))
    e_hat, g_hat = op(OF.fftn(tau), OF.fftn(mu))
    e_ref, g_ref = OF.ifftn(e_hat).real, OF.ifftn(g_hat).real
    dt = torch.float64 if precision == 0 else torch.float32
    e, g = M.mp_green_apply(ctx, precision, n, h, ref, torch.as_tensor(tau, dtype=dt, device="cuda"),
                            torch.as_tensor(mu, dtype=dt, device="cuda"))
    tol = 1e-11 if precision == 0 else 2e-5
    assert np.abs(e.cpu().numpy() - e_ref).max() <= tol * np.abs(e_ref).max()
    assert np.abs(g.cpu().numpy() - g_ref).max() <= tol * np.abs(g_ref).max()


@pytest.mark.parametrize("length", LENGTHS)
@pytest.mark.parametrize("precision", [0, 1])
def test_green_apply_every_line_length(ctx, length, precision):
    if precision == 0 and length > 384:
        pytest.skip("a column of FP64 lines longer than 384 points does not fit a tile")
    _check(ctx, (4, length, 6), precision)
    _check(ctx, (2, 6, length), precision)


@pytest.mark.parametrize("n", [(4, 1, 54), (6, 1, 16), (2, 1, 128), (1, 6, 12), (12, 18, 1), (4, 1, 1)])
@pytest.mark.parametrize("precision", [0, 1])
def test_green_apply_flat_cells(ctx, n, precision):
    _check(ctx, n, precision)


@pytest.mark.parametrize("length", LENGTHS)
@pytest.mark.parametrize("precision", [0, 1])
def test_green_apply_every_row_length(ctx, length, precision):
    """The packed x transforms, several rows per item with the last item cut off."""
    if precision == 0 and length > 324:
        pytest.skip("an FP64 row longer than 324 voxels does not fit pass A's shared memory")
    _check(ctx, (length, 6, 2), precision)
    _check(ctx, (length, 1, 18), precision)
