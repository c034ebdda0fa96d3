"""The performance cases of the micropolar FFT solver: what its users have it do.

A case is one pass through the public entry points of ``paper_2409_10774_gb300``:
whole solves of one cell (``mp_solve``, ``Rve``), batches of cells
(``mp_batch_solve``), a server's requests (``Server``) and the two components
callers use on their own (``mp_green_apply`` / ``mp_green_apply_static`` and
``mp_radial_return``).  Solve outputs are the homogenized results of every
increment and, where the case asks for them, the final fields; those of the
FP32-field precisions are kept in FP32, which is what they hold.  The last
error and the iteration counts say when a solve stopped rather than what it
computed and are left out.

``exact`` evaluates the same problems with plain torch in 64 bits.
"""
import math

import numpy as np
import torch

import paper_2409_10774_gb300 as mp
from paper_2409_10774_gb300.binding import mp_green_apply_static

MATRIX = {"lambda": 20.0, "mu": 12.0, "kappa": 3.0, "alpha": 1.5, "beta": 1.5, "gamma": 1.5,
          "tY": 0.05, "tH": 1.0, "mY": 0.05, "mH": 1.0, "a1": 1.5, "b1": 1.5, "elastic": 0}
INCLUSION = {"lambda": 60.0, "mu": 40.0, "kappa": 10.0, "alpha": 5.0, "beta": 5.0, "gamma": 5.0,
             "tY": 0.0, "tH": 0.0, "mY": 0.0, "mH": 0.0, "a1": 1.5, "b1": 1.5, "elastic": 1}
# material points: perfect plasticity and hardening, with and without a skew couple stress, elastic
POINT_PHASES = [
    dict(MATRIX, alpha=0.0, beta=0.6, mY=0.04, mH=0.7),
    {"lambda": 8.0, "mu": 5.0, "kappa": 2.5, "alpha": 0.9, "beta": 0.2, "gamma": 2.0,
     "tY": 0.03, "tH": 0.0, "mY": 0.02, "mH": 0.0, "a1": 1.2, "b1": 0.8, "elastic": 0},
    dict(MATRIX),
    dict(INCLUSION),
]
REFERENCE = (20.0, 12.0, 3.0, 0.7, 1.1, 1.9)  # reference medium of the Green-operator calls
HOMOGENIZED = ("T", "M", "Eavg", "Gavg", "P", "Q", "Teq", "Meq")
FIELDS = ("e", "g", "t", "m", "p", "q")
# axis lengths the library transforms (1 or even 2^a 3^b), up to 128
LENGTHS = (2, 4, 6, 8, 12, 16, 18, 24, 32, 36, 48, 54, 64, 72, 96, 108, 128)

_context = None


def _ctx():
    """One context per process, as a program keeps it."""
    global _context
    if _context is None:
        _context = mp.Context(0)
    return _context


def listed():
    return [
        # the polycrystal study: a 256^3 cell of 200 grains, device-resident, its first load increments
        {"name": "solve-256", "call": "solve", "resident": True, "precision": 1, "n1": 256, "n2": 256, "n3": 256,
         "cell": "grains", "count": 200, "steps": 2, "of_steps": 9, "tol": 1e-6, "measure": "local", "fields": False},
        # the same study on the largest size of the serving mix, host problem in, homogenized results out
        {"name": "solve-128", "call": "solve", "resident": False, "precision": 1, "n1": 128, "n2": 128, "n3": 128,
         "cell": "grains", "count": 200, "steps": 2, "of_steps": 8, "tol": 1e-6, "measure": "local", "fields": False},
        # a 64^3 regeneration with the all-FP32 level return, loaded through yield
        {"name": "solve-64-fp32-return", "call": "solve", "resident": True, "precision": 2, "n1": 64, "n2": 64,
         "n3": 64, "cell": "grains", "count": 200, "steps": 3, "of_steps": 4, "tol": 1e-6, "measure": "local",
         "fields": False},
        # an uneven box whose lengths have no plan of their own, the averaged error measure
        {"name": "solve-96x54x36", "call": "solve", "resident": False, "precision": 1, "n1": 96, "n2": 54, "n3": 36,
         "cell": "grains", "count": 40, "steps": 3, "of_steps": 6, "tol": 1e-6, "measure": "average",
         "fields": False},
        # the paper's small cell in plain FP64 to a tight tolerance, all fields returned
        {"name": "solve-16-fp64", "call": "solve", "resident": False, "precision": 0, "n1": 16, "n2": 16, "n3": 16,
         "cell": "sphere", "count": 1, "steps": 10, "of_steps": 10, "tol": 1e-8, "measure": "local", "fields": True},
        # the plain FP64 solver on a cell of the batch's largest size
        {"name": "solve-48-fp64", "call": "solve", "resident": True, "precision": 0, "n1": 48, "n2": 48, "n3": 48,
         "cell": "grains", "count": 40, "steps": 2, "of_steps": 8, "tol": 1e-8, "measure": "local", "fields": False},
        # dataset generation: many small cells of uneven sizes in one call
        {"name": "batch-32", "call": "batch", "precision": 1, "cells": 32, "smallest": 16, "largest": 48, "steps": 3,
         "of_steps": 10, "tol": 1e-6},
        # a burst of requests to a running server: stiff inclusions, first increments of their load paths
        {"name": "serve-6", "call": "serve", "precision": 1, "cells": 6, "smallest": 32, "largest": 64, "steps": 2,
         "of_steps": 10, "tol": 1e-6},
        # one application of the Green operator to resident polarization fields, the largest grid
        {"name": "green-256", "call": "green", "static": False, "precision": 1, "n1": 256, "n2": 256, "n3": 256},
        # the allocation-free call inside a latency-critical loop, its largest cube
        {"name": "green-static-48", "call": "green", "static": True, "precision": 1, "n1": 48, "n2": 48, "n3": 48},
        # the material update alone, on the integration points of a large model
        {"name": "return-2m", "call": "return", "precision": 1, "points": 2097152 + 37},
        # ... and on a small one, in FP64: launch and call overhead count
        {"name": "return-5k-fp64", "call": "return", "precision": 0, "points": 5037},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _draw_grid(rng, lo, hi, lengths):
    """Three axis lengths whose product lies in [lo, hi], close to a drawn size."""
    want = _log_uniform(rng, lo, hi)
    while True:
        n = [rng.choice(lengths) for _ in range(3)]
        if rng.random() < 0.4:
            n = [n[0]] * 3
        vox = n[0] * n[1] * n[2]
        if lo <= vox <= hi and 0.5 <= vox / want <= 2.0:
            return n


def draw(rng):
    kind = rng.random()
    if kind < 0.45:  # one cell, every precision, cubes and boxes
        precision = rng.choice((0, 1, 1, 1, 2))
        n = _draw_grid(rng, 512, 96 ** 3 if precision else 48 ** 3, [v for v in LENGTHS if v >= 6])
        vox = n[0] * n[1] * n[2]
        return {"call": "solve", "resident": rng.random() < 0.5, "precision": precision, "n1": n[0], "n2": n[1],
                "n3": n[2], "cell": "grains", "count": rng.randint(5, 200), "steps": rng.randint(1, 4),
                "of_steps": rng.randint(4, 10), "tol": 1e-8 if precision == 0 else 1e-6,
                "measure": rng.choice(("local", "local", "average")), "fields": vox <= 32 ** 3 and rng.random() < 0.5}
    if kind < 0.65:
        return {"call": "batch", "precision": 1, "cells": round(_log_uniform(rng, 2, 64)), "smallest": 16,
                "largest": rng.choice((16, 32, 48)), "steps": rng.randint(1, 3), "of_steps": rng.randint(8, 12),
                "tol": 1e-6}
    if kind < 0.70:
        return {"call": "serve", "precision": 1, "cells": rng.randint(1, 8), "smallest": 32,
                "largest": rng.choice((32, 64)), "steps": rng.randint(1, 2), "of_steps": rng.randint(8, 20),
                "tol": 1e-6}
    if kind < 0.85:
        precision = rng.choice((0, 1, 1))
        static = rng.random() < 0.3
        hi = (32 ** 3 if precision == 0 else 48 ** 3) if static else (96 ** 3 if precision == 0 else 8 * 2 ** 20)
        n = _draw_grid(rng, 64, hi, LENGTHS if static else LENGTHS + (192, 256))
        return {"call": "green", "static": static, "precision": precision, "n1": n[0], "n2": n[1], "n3": n[2]}
    return {"call": "return", "precision": rng.choice((0, 1, 1, 2)), "points": round(_log_uniform(rng, 1000, 3e6))}


# ------------------------------------------------------------------ inputs

def _dist2(n, c):
    """Squared minimum-image distance of every voxel centre (n3, n2, n1) to point c, in voxels."""
    parts = []
    for a in range(3):
        d = torch.arange(n[a], dtype=torch.float32, device="cuda") + (0.5 - float(c[a]))
        d = d - n[a] * torch.round(d / n[a])
        parts.append(d * d)
    return parts[2][:, None, None] + (parts[1][:, None] + parts[0][None, :])[None]


def _grain_map(n, count, rng):
    """Periodic Voronoi tessellation of `count` seeds."""
    best = torch.full((n[2], n[1], n[0]), float("inf"), device="cuda")
    owner = torch.zeros((n[2], n[1], n[0]), dtype=torch.int16, device="cuda")
    for i, c in enumerate(rng.uniform(0.0, 1.0, (count, 3)) * np.array(n)):
        d2 = _dist2(n, c)
        closer = d2 < best
        owner.masked_fill_(closer, i)
        torch.minimum(best, d2, out=best)
    return owner.cpu().numpy().view(np.uint16)


def _sphere_map(n, spheres):
    """Phase 1 inside any of the (centre, radius) spheres, 0 elsewhere."""
    inside = torch.zeros((n[2], n[1], n[0]), dtype=torch.bool, device="cuda")
    for c, r in spheres:
        inside |= _dist2(n, c) <= r * r
    return inside.cpu().numpy().astype(np.uint16)


def _packed_spheres(n, radius, fraction, rng):
    """Random sequential addition of equal non-overlapping periodic spheres."""
    centres = np.empty((0, 3))
    box = np.array(n, dtype=np.float64)
    while len(centres) * 4.0 / 3.0 * math.pi * radius ** 3 < fraction * box.prod():
        c = rng.uniform(0.0, 1.0, 3) * box
        d = c - centres
        d -= box * np.round(d / box)
        if not len(centres) or (d * d).sum(axis=1).min() >= 4.0 * radius * radius:
            centres = np.vstack([centres, c])
    return [(c, radius) for c in centres]


def _ramp(case, E, G):
    """The first `steps` of `of_steps` equal increments of a proportional ramp to (E, G)."""
    frac = np.arange(case["steps"] + 1) / case["of_steps"]
    return frac, frac[:, None, None] * E, frac[:, None, None] * G


def _problem(case, n, phase, phases, E, G, ref_kind):
    time, Ep, Gp = _ramp(case, E, G)
    return {"n": tuple(n), "h": 1.0, "phase": phase, "phases": phases, "time": time, "E": Ep, "G": Gp,
            "tol": case["tol"], "err_kind": case.get("measure", "local"), "ref_kind": ref_kind, "max_iter": 10000}


def _curvature(rng, scale):
    """A mean curvature (bending and torsion) beside the mean strain."""
    return scale * np.array([[0.3, 1.0, 0.0], [0.0, -0.2, 0.0], [-0.5, 0.0, 0.1]]) * rng.uniform(0.8, 1.2)


def _cell_problem(case, seed):
    rng = np.random.default_rng([seed, 1])
    n = (case["n1"], case["n2"], case["n3"])
    if case["cell"] == "sphere":  # one stiff elastic sphere off the grid's centre by less than a voxel
        centre = np.array(n) / 2.0 + rng.uniform(-0.5, 0.5, 3)
        phase = _sphere_map(n, [(centre, min(n) / 4.0)])
        E = np.diag([0.005, 0.0, 0.0]) * rng.uniform(0.98, 1.02)
        return _problem(case, n, phase, [MATRIX, INCLUSION], E, _curvature(rng, 0.0005), "midrange")
    rows = []
    for _ in range(case["count"]):  # moduli and yield stresses within 20 % of the matrix's
        row = dict(MATRIX)
        for key in ("lambda", "mu", "kappa", "alpha", "beta", "gamma", "tY", "mY"):
            row[key] = MATRIX[key] * rng.uniform(0.8, 1.2)
        row["beta"] = min(row["beta"], row["gamma"])
        rows.append(row)
    E = np.array([[0.01, 0.003, 0.0], [0.0, 0.0, 0.001], [0.0, 0.0, -0.002]]) * rng.uniform(0.98, 1.02)
    return _problem(case, n, _grain_map(n, case["count"], rng), rows, E, _curvature(rng, 0.001), "mean")


def _many_problems(case, seed):
    """Cells of a batch (overlapping spheres, a drawn intrinsic length) or of a
    server's queue (packed spheres ten times as stiff as the matrix)."""
    rng = np.random.default_rng([seed, 2])
    sizes = [v for v in ((16, 24, 32, 48) if case["call"] == "batch" else (32, 48, 64))
             if case["smallest"] <= v <= case["largest"]]
    out = []
    for i in range(case["cells"]):
        n = (sizes[i % len(sizes)],) * 3
        E = rng.standard_normal((3, 3))
        E *= 0.005 / np.linalg.norm(E)
        if case["call"] == "batch":
            spheres = [(rng.uniform(0.0, 1.0, 3) * np.array(n), rng.uniform(3.0, 8.0))
                       for _ in range(rng.integers(1, 9))]
            length = math.exp(rng.uniform(math.log(0.1), math.log(10.0)))
            rows = [dict(r, alpha=r["mu"] * length ** 2, beta=r["mu"] * length ** 2, gamma=r["mu"] * length ** 2)
                    for r in (MATRIX, INCLUSION)]
            G = _curvature(rng, 0.0005 / max(1.0, length) ** 2)  # the couple stresses stay of one size
        else:
            spheres = _packed_spheres(n, 6.0, 0.25, rng)
            stiff = {k: 10.0 * MATRIX[k] for k in ("lambda", "mu", "kappa", "alpha", "beta", "gamma")}
            rows = [MATRIX, dict(MATRIX, **stiff, elastic=1)]
            G = _curvature(rng, 0.0005)
        out.append(_problem(case, n, _sphere_map(n, spheres), rows, E, G, "midrange"))
    return out


def _points(case, seed):
    """Material-point states around the yield surfaces, most of them moving plastically."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    count = case["points"]
    real = torch.float64 if case["precision"] == 0 else torch.float32

    def normal(scale):
        return scale * torch.randn((count, 3, 3), generator=gen, device="cuda", dtype=torch.float64)

    pid = torch.randint(0, len(POINT_PHASES), (count,), generator=gen, device="cuda")
    size = 10.0 ** (torch.rand((count, 1, 1), generator=gen, device="cuda", dtype=torch.float64) * 1.5 - 1.2)
    e, g = normal(0.002), normal(0.002)
    e_n, g_n = e + normal(0.0006), g + normal(0.0006)
    t_n, m_n = normal(0.02), normal(0.02)
    # a history where gamma == beta has a symmetric couple stress
    even = torch.tensor([r["gamma"] == r["beta"] for r in POINT_PHASES], device="cuda")[pid][:, None, None]
    m_n = torch.where(even, 0.5 * (m_n + m_n.transpose(1, 2)), m_n)
    tensors = [(x * size).to(real).contiguous() for x in (e, g, e_n, g_n, t_n, m_n)]
    p_n, q_n = (0.01 * torch.rand(count, generator=gen, device="cuda", dtype=torch.float64) for _ in range(2))
    return [pid.to(torch.int16)] + tensors + [p_n, q_n]


def _polarization(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    shape = (case["n3"], case["n2"], case["n1"], 3, 3)
    real = torch.float64 if case["precision"] == 0 else torch.float32
    return [0.05 * torch.randn(shape, generator=gen, device="cuda", dtype=real) for _ in range(2)]


def prepare(case, seed):
    state = {"case": case, "ctx": _ctx()}
    if case["call"] == "solve":
        state["problem"] = _cell_problem(case, seed)
        if case["resident"]:
            state["cell"] = mp.Rve(state["ctx"], state["problem"], precision=case["precision"])
    elif case["call"] in ("batch", "serve"):
        state["problems"] = _many_problems(case, seed)
        if case["call"] == "serve":
            state["server"] = mp.Server(state["ctx"], budget_bytes=4 << 30)
    elif case["call"] == "green":
        state["fields"] = _polarization(case, seed)
        if case["static"]:
            state["out"] = [torch.empty_like(x) for x in state["fields"]]
    else:
        state["points"] = _points(case, seed)
    return state


# ------------------------------------------------------------------ the passes

def _results(case, res):
    real = np.float64 if case["precision"] == 0 else np.float32
    out = {k: res[k].astype(real) for k in HOMOGENIZED}
    if case.get("fields"):
        out.update({"field_" + k: res["final"][k].astype(real) for k in FIELDS})
    return out


def _stacked(results):
    """One array per quantity over the cells of a call (they have equally many increments)."""
    return {k: np.stack([r[k] for r in results]) for k in results[0]}


def run(state):
    case, ctx = state["case"], state["ctx"]
    precision = case["precision"]
    if case["call"] == "solve":
        if case["resident"]:
            cell = state["cell"]
            cell.reset()
            cell.run(case["steps"])
            return _results(case, cell.results(fields=case["fields"]))
        return _results(case, mp.mp_solve(ctx, state["problem"], precision=precision, fields=case["fields"]))
    if case["call"] == "batch":
        return _stacked([_results(case, r) for r in mp.mp_batch_solve(ctx, state["problems"], precision=precision)])
    if case["call"] == "serve":
        server = state["server"]
        tickets = [server.submit(p, precision=precision) for p in state["problems"]]
        return _stacked([_results(case, server.wait(t)) for t in tickets])
    if case["call"] == "green":
        n = (case["n1"], case["n2"], case["n3"])
        if case["static"]:
            return mp_green_apply_static(ctx, precision, n, 1.0, REFERENCE, *state["fields"], *state["out"])
        return mp.mp_green_apply(ctx, precision, n, 1.0, REFERENCE, *state["fields"])
    phase, *rest = state["points"]
    return mp.mp_radial_return(ctx, precision, phase, POINT_PHASES, *rest)


def work(case):
    """Bytes and operations of one pass.  A fixed-point iteration reads and
    writes the half spectrum twice (y-z operator, x transforms), reads and
    writes the iterate, and reads the history and the plastic strains; it
    transforms 18 real fields both ways, applies the operator (~230 operations
    per half-spectrum point) and the material update (~700 per voxel with the
    polarization and the error norms).  Iterations per increment are typical
    ones; those of a polycrystal's elastic first increment are few."""
    size = 8 if case["precision"] == 0 else 4
    if case["call"] == "return":
        return {"bytes": case["points"] * (8 * 9 * size + 2 + 4 * 8), "flops": case["points"] * 400}
    if case["call"] == "green":
        vox = case["n1"] * case["n2"] * case["n3"]
        return {"bytes": 36 * size * vox, "flops": vox * (18 * 5 * math.log2(max(vox, 2)) + 115)}
    if case["call"] == "solve":
        cells = [case["n1"] * case["n2"] * case["n3"]]
        iters = 9 + 55 * (case["steps"] - 1) if case["cell"] == "grains" else 90 * case["steps"]
    else:
        sizes = [v for v in ((16, 24, 32, 48) if case["call"] == "batch" else (32, 48, 64))
                 if case["smallest"] <= v <= case["largest"]]
        cells = [sizes[i % len(sizes)] ** 3 for i in range(case["cells"])]
        iters = 75 * case["steps"]
    vox = sum(cells)
    flops = 18 * 5 * math.log2(max(vox / len(cells), 2)) + 115 + 700
    return {"bytes": vox * iters * ((72 + 60) * size + 16), "flops": vox * iters * flops}


# ------------------------------------------------------------------ 64-bit values

def _contract(a, b, lam, x):
    """a x_kl + b x_lk + lam tr(x) d_kl"""
    tr = x.diagonal(dim1=-2, dim2=-1).sum(-1)
    eye = torch.eye(3, dtype=x.dtype, device=x.device)
    return a * x + b * x.transpose(-1, -2) + (lam * tr[..., None, None]) * eye


def _table(phases, pid):
    """Per-point material parameters, shaped to scale tensors."""
    rows = {k: torch.tensor([float(r[k]) for r in phases], dtype=torch.float64, device="cuda")[pid]
            for k in MATRIX}
    return {k: v[..., None, None] for k, v in rows.items()}


def _stress(P, x):
    return _contract(P["mu"] + P["kappa"], P["mu"] - P["kappa"], P["lambda"], x)


def _couple(P, x):
    return _contract(P["beta"], P["gamma"], P["alpha"], x)


def _material(P, ht, hm, e, g, p, q):
    """Trial stresses from the history, scaled back to the yield surfaces."""
    t, m = ht + _stress(P, e), hm + _couple(P, g)
    eye = torch.eye(3, dtype=t.dtype, device=t.device)
    vol = t.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None] / 3.0 * eye
    plastic = P["elastic"] == 0

    def level(s, c_sym, c_skw, hard, yld, modulus, acc):
        sym, skw = 0.5 * (s + s.transpose(-1, -2)), 0.5 * (s - s.transpose(-1, -2))
        eq = torch.sqrt(c_sym * (sym * sym).sum((-1, -2), keepdim=True)
                        + c_skw * (skw * skw).sum((-1, -2), keepdim=True))
        radius = yld + hard * acc
        step = torch.where(plastic & (eq >= radius), (eq - radius) / (hard + modulus), torch.zeros_like(eq))
        return torch.where(step > 0, 1.0 - modulus * step / eq, torch.ones_like(eq)), acc + step

    gap = P["gamma"] - P["beta"]
    both = P["gamma"] + P["beta"]
    b2 = torch.where(gap > 0, P["b1"] * both / gap, torch.zeros_like(gap))
    ft, p = level(t - vol, P["a1"], P["a1"] * P["mu"] / P["kappa"], P["tH"], P["tY"],
                  2.0 * P["a1"] * P["mu"], p)
    fm, q = level(m, P["b1"], b2, P["mH"], P["mY"], P["b1"] * both, q)
    return vol + ft * (t - vol), fm * m, p, q


def _equivalent(P, t, m):
    dev = t - t.diagonal(dim1=-2, dim2=-1).mean(-1)[..., None, None] * torch.eye(3, dtype=t.dtype, device=t.device)

    def norm(s, c_sym, c_skw):
        sym, skw = 0.5 * (s + s.transpose(-1, -2)), 0.5 * (s - s.transpose(-1, -2))
        return torch.sqrt((c_sym * sym * sym + c_skw * skw * skw).sum((-1, -2)))

    gap = P["gamma"] - P["beta"]
    b2 = torch.where(gap > 0, P["b1"] * (P["gamma"] + P["beta"]) / gap, torch.zeros_like(gap))
    return norm(dev, P["a1"], P["a1"] * P["mu"] / P["kappa"]), norm(m, P["b1"], b2)


def _operator(n, h, ref):
    """Applies the reference medium's Green operator to (tau, mu): per
    wavevector, the balance of force and moment solved for the displacement u
    and rotation phi, and their strain and curvature."""
    lam, mu, kap, al, be, ga = (float(v) for v in ref)
    freq = [2.0 * math.pi * np.fft.fftfreq(k) for k in n]
    axes = [torch.tensor(f[: k // 2 + 1] if a == 0 else f, device="cuda") for a, (f, k) in enumerate(zip(freq, n))]
    keep = [torch.tensor([not (k % 2 == 0 and i == k // 2) for i in range(len(ax))], device="cuda")
            for k, ax in zip(n, axes)]
    live = keep[2][:, None, None] & keep[1][None, :, None] & keep[0][None, None, :]
    x = [(axes[0] / h)[None, None, :], (axes[1] / h)[None, :, None], (axes[2] / h)[:, None, None]]
    x[0] = x[0].abs()
    k2 = x[0] ** 2 + x[1] ** 2 + x[2] ** 2
    live = live & (k2 > 0)
    k2 = torch.where(live, k2, torch.ones_like(k2))
    on = live.to(torch.float64)
    a, b = (mu + kap) * k2, ga * k2 + 4.0 * kap
    inv = on / (k2 * ((mu + kap) * ga * k2 + 4.0 * kap * mu))
    along_u, along_p = on / (k2 * k2 * (lam + 2.0 * mu)), on / (k2 * ((al + be + ga) * k2 + 4.0 * kap))

    def dot(v):
        return x[0] * v[0] + x[1] * v[1] + x[2] * v[2]

    def cross(v):
        return [x[1] * v[2] - x[2] * v[1], x[2] * v[0] - x[0] * v[2], x[0] * v[1] - x[1] * v[0]]

    def forward(v):
        return torch.fft.rfftn(v, dim=(0, 1, 2))

    def back(v):
        return torch.fft.irfftn(v, s=(n[2], n[1], n[0]), dim=(0, 1, 2))

    def apply(tau, mom):
        f, g = [], []
        for l in range(3):
            f.append(0)
            g.append(0)
            for k in range(3):
                f[l] = f[l] + 1j * x[k] * forward(tau[..., k, l])
                g[l] = g[l] + 1j * x[k] * forward(mom[..., k, l])
            r, s = (l + 1) % 3, (l + 2) % 3
            g[l] = g[l] + forward(tau[..., r, s] - tau[..., s, r])
        xf, xg, cf, cg = dot(f), dot(g), cross(f), cross(g)
        u = [x[l] * xf * along_u + (b * (f[l] - x[l] * xf / k2) + 2j * kap * cg[l]) * inv for l in range(3)]
        w = [x[l] * xg * along_p + (a * (g[l] - x[l] * xg / k2) + 2j * kap * cf[l]) * inv for l in range(3)]
        e, c = torch.empty_like(tau), torch.empty_like(mom)
        for k in range(3):
            for l in range(3):
                v = 1j * x[k] * u[l]
                if k != l:  # eps_lkm phi_m
                    m = 3 - k - l
                    v = v + (w[m] if (l, k, m) in ((0, 1, 2), (1, 2, 0), (2, 0, 1)) else -w[m])
                e[..., k, l] = back(v)
                c[..., k, l] = back(1j * x[l] * w[k])
        return e, c

    return apply


def _solve64(case, problem):
    """The increments' equilibrium fields, iterated well below the case's tolerance."""
    n = problem["n"]
    pid = torch.tensor(problem["phase"].astype(np.int64), device="cuda").reshape(n[2], n[1], n[0])
    rows = problem["phases"]
    P = _table(rows, pid)
    present = np.bincount(problem["phase"].reshape(-1), minlength=len(rows))
    moduli = np.array([[r[k] for k in ("lambda", "mu", "kappa", "alpha", "beta", "gamma")] for r in rows])
    if problem["ref_kind"] == "mean":
        ref = (moduli * present[:, None]).sum(axis=0) / present.sum()
    else:
        seen = moduli[present > 0]
        ref = 0.5 * (seen.min(axis=0) + seen.max(axis=0))
    P0 = {k: float(v) for k, v in zip(("lambda", "mu", "kappa", "alpha", "beta", "gamma"), ref)}
    apply = _operator(n, problem["h"], ref)
    zero = torch.zeros(tuple(pid.shape) + (3, 3), dtype=torch.float64, device="cuda")
    ht, hm, e, g = zero, zero, zero, zero
    old = (zero, zero)
    p = q = zero[..., :1, :1]
    out = {k: [] for k in HOMOGENIZED}
    for s in range(1, case["steps"] + 1):
        E, G = (torch.tensor(problem[k][s], device="cuda") for k in ("E", "G"))
        # equal increments: linear extrapolation of the last two converged states
        start = (E + zero, G + zero) if s == 1 else (2.0 * e - old[0], 2.0 * g - old[1])
        old = (e, g)
        e, g = start
        size = max(float(E.norm()), problem["h"] * float(G.norm()))
        best, since = math.inf, 0
        for it in range(6000):
            t, m, _, _ = _material(P, ht, hm, e, g, p, q)
            de, dg = apply(t - _stress_ref(P0, e), m - _couple_ref(P0, g))
            e_new, g_new = E + de, G + dg
            if it % 4 == 3:
                err = max(float((e_new - e).abs().max()), problem["h"] * float((g_new - g).abs().max())) / size
                best, since = (err, 0) if err < 0.9 * best else (best, since + 1)
                if err <= 0.02 * case["tol"] or since > 100:
                    e, g = e_new, g_new
                    break
            e, g = e_new, g_new
        t, m, p, q = _material(P, ht, hm, e, g, p, q)
        ht, hm = t - _stress(P, e), m - _couple(P, g)
        teq, meq = _equivalent(P, t, m)
        for key, v in zip(HOMOGENIZED, (t, m, e, g)):
            out[key].append(v.mean((0, 1, 2)))
        for key, v in zip(HOMOGENIZED[4:], (p, q, teq, meq)):
            out[key].append(v.mean())
    res = {k: torch.stack(v).cpu().numpy() for k, v in out.items()}
    if case.get("fields"):
        for key, v in zip(FIELDS, (e, g, t, m, p[..., 0, 0], q[..., 0, 0])):
            res["field_" + key] = v.cpu().numpy()
    return res


def _stress_ref(P, x):
    return _contract(P["mu"] + P["kappa"], P["mu"] - P["kappa"], P["lambda"], x)


def _couple_ref(P, x):
    return _contract(P["beta"], P["gamma"], P["alpha"], x)


def exact(case, seed):
    if case["call"] == "solve":
        return _solve64(case, _cell_problem(case, seed))
    if case["call"] in ("batch", "serve"):
        return _stacked([_solve64(case, p) for p in _many_problems(case, seed)])
    if case["call"] == "green":
        tau, mom = (x.double() for x in _polarization(case, seed))
        return _operator((case["n1"], case["n2"], case["n3"]), 1.0, REFERENCE)(tau, mom)
    pid, e, g, e_n, g_n, t_n, m_n, p_n, q_n = _points(case, seed)
    P = _table(POINT_PHASES, pid.long())
    e, g, e_n, g_n, t_n, m_n = (x.double() for x in (e, g, e_n, g_n, t_n, m_n))
    t, m, p, q = _material(P, t_n - _stress(P, e_n), m_n - _couple(P, g_n), e, g, p_n[:, None, None],
                           q_n[:, None, None])
    return t, m, p[:, 0, 0], q[:, 0, 0]
