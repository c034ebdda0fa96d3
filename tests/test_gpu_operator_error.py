"""The FP32 Green operator's distance from its FP64 value on random fields.

Each entry is the distance (root mean square over e and gamma, relative, mean
of four seeds) of the kernels whose sums of products are fused and whose
transforms carry all 18 fields: the rounding a faster form must not exceed.
The seeds differ by 0.3 % of it; the flat cells' kernels, which do the same
operations in other orders, are allowed 1 %, the boxes' nothing.  The FP64
operator serves as the value (6e-16, test_gpu_line_lengths.py holds it to the
oracle).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

REFERENCE = (20.0, 12.0, 3.0, 0.7, 1.1, 1.9)


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2409_10774_gb300 as M
    return M.Context(0)


def _distance(ctx, n):
    import paper_2409_10774_gb300 as M
    per_seed = []
    for seed in range(4):
        rng = np.random.default_rng([seed, *n])
        shape = (n[2], n[1], n[0], 3, 3)
        tau, mu = (torch.as_tensor(rng.standard_normal(shape).astype(np.float32), device="cuda") for _ in range(2))
        f32 = M.mp_green_apply(ctx, 1, n, 0.83, REFERENCE, tau, mu)
        f64 = M.mp_green_apply(ctx, 0, n, 0.83, REFERENCE, tau.double(), mu.double())
        rel = [float((a.double() - b).norm() / b.norm()) for a, b in zip(f32, f64)]
        per_seed.append(np.sqrt(np.mean(np.square(rel))))
    return float(np.mean(per_seed))


# cells without a y pass: the z pass transforms all 18 fields
@pytest.mark.parametrize("n, bound", [((64, 1, 64), 2.011e-7), ((128, 1, 128), 2.125e-7)])
def test_flat_cells(ctx, n, bound):
    assert _distance(ctx, n) <= 1.01 * bound


# boxes: the z pass transforms the reduced fields
@pytest.mark.parametrize("n, bound", [((16, 16, 16), 1.871e-7), ((32, 32, 32), 2.302e-7), ((64, 64, 64), 2.462e-7),
                                      ((96, 54, 36), 2.717e-7), ((24, 18, 72), 2.555e-7)])
def test_boxes(ctx, n, bound):
    assert _distance(ctx, n) <= bound
