"""Algorithm 1 on material points at the edges of its launch rules, against the
oracle: chunk remainders, small and large calls, arrays that start off a
16-byte boundary, and phase tables that do not fit the launch arguments.
Tolerances as in test_gpu_parity.py (FP64 1e-12, FP32 2e-6 relative).
"""
import numpy as np
import pytest

import workloads as W
from oracle import constitutive as OC

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2409_10774_gb300 as M
    return M.Context(0)


def _phases(count):
    rng = np.random.default_rng(count)
    rows = []
    for k in range(count):
        row = dict(W.generators._matrix_row(rng.uniform(0.5, 3.0)))
        row["beta"] = row["gamma"] * rng.choice((0.4, 1.0))
        row["elastic"] = int(k % 5 == 4)
        rows.append(row)
    return W.phase_record(rows)


@pytest.mark.parametrize("count,n_phases,offset", [
    (1, 1, 0), (31, 3, 0), (33, 3, 1), (128, 12, 0), (129, 13, 0), (4999, 12, 3), (40001, 3, 0), (40001, 40, 1)])
@pytest.mark.parametrize("precision", [0, 1])
def test_radial_return_edges(ctx, count, n_phases, offset, precision):
    import paper_2409_10774_gb300 as M
    phases = _phases(n_phases)
    rng = np.random.default_rng(count + n_phases)
    pid = rng.integers(0, n_phases, count).astype(np.uint16)
    s = W.random_material_states(count, count, strain_scale=0.002, history_scale=0.02, p_scale=0.01)
    f = 10.0 ** rng.uniform(-1.2, 0.3, count)
    for k in ("e", "g", "e_n", "g_n", "t_n", "m_n"):
        s[k] = s[k] * f[:, None, None]
    even = phases["gamma"][pid] == phases["beta"][pid]
    s["m_n"][even] = OC.sym(s["m_n"][even])
    want = [np.empty_like(s["e"]), np.empty_like(s["e"]), np.empty(count), np.empty(count)]
    for k in range(n_phases):
        i = pid == k
        if i.any():
            res = OC.radial_return(*(s[a][i] for a in ("e", "g", "e_n", "g_n", "t_n", "m_n", "p_n", "q_n")), phases[k])
            for w, r in zip(want, res):
                w[i] = r
    real = torch.float64 if precision == 0 else torch.float32

    def dev(a, dtype=real):
        # `offset` elements into a larger array: contiguous, off the 16-byte boundary
        a = torch.as_tensor(np.ascontiguousarray(a)).to(dtype)
        big = torch.zeros(a.numel() + offset, dtype=dtype, device="cuda")
        big[offset:] = a.reshape(-1).cuda()
        return big[offset:].view(a.shape)

    got = M.mp_radial_return(ctx, precision, dev(pid.astype(np.int16), torch.int16), phases,
                             *(dev(s[a]) for a in ("e", "g", "e_n", "g_n", "t_n", "m_n")),
                             *(dev(s[a], torch.float64) for a in ("p_n", "q_n")))
    tol = 1e-12 if precision == 0 else 2e-6
    for g, w in zip(got, want):
        assert np.abs(g.cpu().numpy() - w).max() <= tol * np.abs(w).max()
