"""The workloads whose speed this library is held to.

Each case is one call, or one short sequence of calls, that a program using the
library repeats, through the public binding and with the problem families, sizes
and options of the repository's tests, benchmark and documentation:

- ``system``: one linear system of an outer method the caller wrote itself:
  ``kkt_assemble`` with new D (and W), ``kkt_factor``, ``kkt_solve``;
- ``solve``: more right-hand sides against a factor that is already held;
- ``direction``: one Newton direction (``ipm_newton_direction``) from an iterate;
- ``ipm``: a whole cold-start LP solve (``ipm_solve``);
- ``mpc``: a whole batch of small MPC QPs (``BatchedMPC.ipm_solve_batched``).

The symbolic analysis and the workspace are made once per pattern by every
program (they are part of ``prepare``); J, W, D, the iterate and the right-hand
sides change from call to call, so they are drawn anew for every seed.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import gen
import paper_2508_16094_gb300 as gb

PREC = {"fp64": gb.IPM_FP64, "fp64_tc": gb.IPM_FP64, "fp32": gb.IPM_FP32, "tf32": gb.IPM_TF32,
        "tf32x3": gb.IPM_TF32X3, "bf16": gb.IPM_BF16}
FORM = {"primal": gb.IPM_FORM_PRIMAL, "augmented": gb.IPM_FORM_AUGMENTED}
REG = 1e-8  # delta_p and delta_d, the defaults
LOWER, UPPER = 0.0, 10.0  # bounds of the LP families


def listed():
    grid = lambda x, y, z: {"family": "grid", "x": x, "y": y, "z": z}
    return [
        # the small random LP (2000 variables, 1000 rows), solved from a cold start in the
        # default arithmetic: many short launches, the latency of one iteration is what counts
        {"name": "ipm_random2000_fp64", "kind": "ipm", "family": "random", "n": 2000, "m": 1000,
         "prec": "fp64", "tol": 1e-6},
        # a small structured system, one of thousands in a sequence: nothing but latency
        {"name": "system_grid10_tf32x3", "kind": "system", **grid(10, 10, 10), "prec": "tf32x3",
         "qp": False, "decades": 1.0},
        # the default arithmetic (FP64 throughout) at an ordinary size
        {"name": "system_grid32_fp64", "kind": "system", **grid(32, 32, 32), "prec": "fp64",
         "qp": False, "decades": 1.0},
        # the same accuracy with the updates on the tensor cores
        {"name": "system_grid40_fp64tc", "kind": "system", **grid(40, 40, 40), "prec": "fp64_tc",
         "qp": False, "decades": 1.0},
        # the recommended mixed precision at the size the benchmark compares all forms on
        {"name": "system_grid48_tf32x3", "kind": "system", **grid(48, 48, 48), "prec": "tf32x3",
         "qp": False, "decades": 1.0},
        # the largest factor here, in the cheapest arithmetic of a ladder's first rungs; a QP
        {"name": "system_grid64_tf32_qp", "kind": "system", **grid(64, 64, 64), "prec": "tf32",
         "qp": True, "decades": 1.0},
        # several right-hand sides against one held FP64 factor (sensitivities, multiple targets)
        {"name": "solve_grid40_fp64_rhs4", "kind": "solve", **grid(40, 40, 40), "prec": "fp64_tc",
         "qp": False, "decades": 1.0, "nrhs": 4},
        # ... and against a mixed-precision factor, each refined to FP64 accuracy
        {"name": "solve_grid56_tf32x3_rhs8", "kind": "solve", **grid(56, 56, 56), "prec": "tf32x3",
         "qp": False, "decades": 1.0, "nrhs": 8},
        # one step of the method on a box that is no power of two in any direction
        {"name": "direction_grid23x41x18_tf32x3", "kind": "direction", **grid(23, 41, 18),
         "prec": "tf32x3", "form": "primal", "decades": 1.0},
        # the same through the augmented system (signed pivot-free LDL^T, FP64)
        {"name": "direction_grid11x12x13_augmented", "kind": "direction", **grid(11, 12, 13),
         "prec": "fp64", "form": "augmented", "decades": 1.0},
        # a controller's worth of MPC problems, and the full batch
        {"name": "mpc_96", "kind": "mpc", "count": 96, "t_min": 10, "t_max": 100},
        {"name": "mpc_4096", "kind": "mpc", "count": 4096, "t_min": 10, "t_max": 100},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, points_lo, points_hi, side_hi):
    """Sides of a box with about a log-uniform number of points; sides within a factor of two."""
    while True:
        p = math.exp(rng.uniform(math.log(points_lo), math.log(points_hi)))
        a, b = rng.uniform(-0.3, 0.3), rng.uniform(-0.3, 0.3)
        s = p ** (1.0 / 3.0)
        x, y, z = (max(2, int(round(s * math.exp(t)))) for t in (a, b, -a - b))
        if points_lo <= x * y * z <= points_hi and max(x, y, z) <= side_hi:
            return {"family": "grid", "x": x, "y": y, "z": z}


def draw(rng):
    kind = rng.choice(["ipm", "system", "system", "system", "solve", "solve", "direction", "mpc"])
    if kind == "ipm":
        n = _log_int(rng, 300, 2000)
        return {"kind": kind, "family": "random", "n": n, "m": n // 2, "prec": "fp64", "tol": 1e-6}
    if kind == "mpc":
        lo = rng.randint(2, 40)
        return {"kind": kind, "count": _log_int(rng, 16, 4000), "t_min": lo, "t_max": lo + rng.randint(0, 55)}
    if kind == "direction":
        form = rng.choice(["primal", "primal", "augmented"])
        prec = "fp64" if form == "augmented" else rng.choice(["fp64", "tf32x3", "tf32x3"])
        hi = 2000 if form == "augmented" else 25000
        return {"kind": kind, **_box(rng, 500, hi, 60), "prec": prec, "form": form, "decades": 1.0}
    prec = rng.choice(["fp64", "fp64_tc", "tf32x3", "tf32x3", "tf32", "bf16", "fp32"])
    if kind == "system":
        hi = {"fp64": 30000, "fp64_tc": 60000, "fp32": 60000}.get(prec, 200000)
        return {"kind": kind, **_box(rng, 300, hi, 90), "prec": prec, "qp": rng.random() < 0.3,
                "decades": round(rng.uniform(0.3, 1.0), 2)}
    prec = {"fp64": "fp64_tc", "bf16": "tf32x3"}.get(prec, prec)
    hi = {"fp64_tc": 60000, "fp32": 60000}.get(prec, 150000)
    return {"kind": kind, **_box(rng, 2000, hi, 80), "prec": prec, "qp": rng.random() < 0.3,
            "decades": round(rng.uniform(0.3, 1.0), 2), "nrhs": rng.randint(1, 8)}


# ---- patterns (one per size, whatever the seed) -------------------------------
@functools.lru_cache(maxsize=4)
def _grid_pattern(x, y, z):
    lp = gen.grid_lp(x, y, z, seed=1)
    rows = np.repeat(np.arange(lp.m), np.diff(lp.rowptr))
    return lp.n, lp.m, lp.rowptr, lp.col, np.flatnonzero(lp.col == rows), gen.nd_order_grid3d(x, y, z)


@functools.lru_cache(maxsize=4)
def _random_pattern(n, m):
    lp = gen.random_lp(n, m, 5, seed=0)
    return lp.n, lp.m, lp.rowptr, lp.col, np.zeros(0, np.int64), gen.lp_ordering(lp, "md")


def _pattern(case):
    if case["family"] == "grid":
        return _grid_pattern(case["x"], case["y"], case["z"])
    return _random_pattern(case["n"], case["m"])


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, count, lo, hi):
    return lo + (hi - lo) * torch.rand(count, generator=g, dtype=torch.float64, device="cuda")


class _Sparse:
    """Plain torch products with J (m x n, CSR) and its transpose."""

    def __init__(self, n, m, rowptr, col, val):
        dev = lambda a: torch.as_tensor(a, device="cuda")
        idx = torch.stack([dev(np.repeat(np.arange(m), np.diff(rowptr))), dev(col).long()])
        J = torch.sparse_coo_tensor(idx, val, (m, n)).coalesce()
        self.J, self.JT = J.to_sparse_csr(), J.t().coalesce().to_sparse_csr()

    def mul(self, v):
        return (self.J @ v.unsqueeze(1)).squeeze(1)

    def tmul(self, v):
        return (self.JT @ v.unsqueeze(1)).squeeze(1)


def _problem(case, seed):
    """Problem data of the grid and random LP families, drawn on the GPU."""
    n, m, rowptr, col, diag, _ = _pattern(case)
    g = _generator(seed)
    val = torch.randn(len(col), generator=g, dtype=torch.float64, device="cuda")
    if len(diag):
        val[torch.as_tensor(diag, device="cuda")] += 8.0
    d = {"n": n, "m": m, "mt": m + 2 * n, "val": val, "g": g, "w": None}
    if case.get("qp"):
        d["w"] = _uniform(g, n, 0.1, 10.0)  # a diagonal Hessian
    return d


def _context(case, **options):
    n, m, rowptr, col, _, perm = _pattern(case)
    l, u = np.full(n, LOWER), np.full(n, UPPER)
    wp, wi = (np.arange(n + 1), np.arange(n)) if case.get("qp") else (None, None)
    prec = PREC[case["prec"]]
    o = gb.default_options(precision=prec, storage_fp64=int(prec == gb.IPM_FP64),
                           fp64_tc=int(case["prec"] == "fp64_tc"), **options)
    ctx = gb.IpmContext(n, m, rowptr, col, l, u, wp, wi, options=o)
    ctx.kkt_analyze(_augmented_order(perm, m) if case.get("form") == "augmented" else perm)
    ctx.ipm_set_workspace()
    return ctx


def _augmented_order(perm, m):
    """Each row's multiplier right after the variable of the same grid point."""
    return np.stack([perm, len(perm) + perm], 1).ravel().astype(np.int32) if m == len(perm) else None


def _system_data(case, seed):
    d = _problem(case, seed)
    d["D"] = 10.0 ** _uniform(d["g"], d["mt"], -case["decades"], case["decades"])
    k = case.get("nrhs", 1)
    d["rhs"] = torch.randn(k, d["n"], generator=d["g"], dtype=torch.float64, device="cuda")
    return d


def _direction_data(case, seed):
    """An iterate inside its bounds, s and lambda off the central path by some decades."""
    d = _problem(case, seed)
    n, m, rowptr, col, _, _ = _pattern(case)
    g, e = d["g"], case["decades"]
    d["x"] = _uniform(g, n, LOWER + 1.0, UPPER - 1.0)
    J = _Sparse(n, m, rowptr, col, d["val"])
    d["b"] = J.mul(d["x"]) - _uniform(g, m, 0.1, 1.0)
    d["c"] = J.tmul(_uniform(g, m, 0.0, 1.0)) + _uniform(g, n, 0.1, 1.0)
    d["s"] = 10.0 ** _uniform(g, d["mt"], -0.5 * e, 0.5 * e)
    d["lam"] = 10.0 ** _uniform(g, d["mt"], -0.5 * e, 0.5 * e)
    d["target"] = torch.full((d["mt"],), 0.1, dtype=torch.float64, device="cuda")
    return d


def _ipm_data(case, seed):
    d = _problem(case, seed)
    n, m, rowptr, col, _, _ = _pattern(case)
    g = d["g"]
    J = _Sparse(n, m, rowptr, col, d["val"])
    d["b"] = J.mul(_uniform(g, n, 1.0, 9.0)) - _uniform(g, m, 0.1, 1.0)
    d["c"] = J.tmul(_uniform(g, m, 0.0, 1.0)) + _uniform(g, n, 0.1, 1.0)
    return d


class _Mpc:
    """Arrays as BatchedMPC takes them."""


def _mpc_data(case, seed):
    """The recipe of gen.mpc_batch, drawn for all instances at once: A_k scaled to spectral
    radius 0.95 (from the norm of its 2^12-th power), x_0 redrawn until the trajectory with
    u = 0 stays inside the box."""
    count, g = case["count"], _generator(seed)
    f64 = dict(dtype=torch.float64, device="cuda")
    # the horizons belong to the controllers, not to the moment
    T = torch.as_tensor(gen.uniform(7, count, case["t_min"], case["t_max"] + 1).astype(np.int32), device="cuda").long()
    stages = int(T.sum())
    G = torch.randn(stages, 12, 12, generator=g, **f64)
    P, log = G.clone(), torch.zeros(stages, **f64)
    for k in range(12):
        norm = torch.linalg.matrix_norm(P)
        log += torch.log(norm) / 2.0 ** k
        P = P / norm[:, None, None]
        P = P @ P
    A = 0.95 * G / torch.exp(log + torch.log(torch.linalg.matrix_norm(P)) / 2.0 ** 12)[:, None, None]
    B = torch.randn(stages, 12, 4, generator=g, **f64)
    Q = 0.1 + 9.9 * torch.rand(count, 12, generator=g, **f64)
    R = 0.1 + 9.9 * torch.rand(count, 4, generator=g, **f64)
    off = torch.cumsum(T, 0) - T
    x0 = torch.zeros(count, 12, **f64)
    todo, scale = torch.ones(count, dtype=torch.bool, device="cuda"), 1.0
    for _ in range(60):
        cand = scale * (2.0 * torch.rand(count, 12, generator=g, **f64) - 1.0)
        x, ok = cand, todo.clone()
        for k in range(int(T.max())):
            on = k < T
            x = torch.where(on[:, None], (A[torch.where(on, off + k, 0)] @ x[:, :, None])[:, :, 0], x)
            ok &= x.abs().amax(1) <= 5.0
        x0 = torch.where(ok[:, None], cand, x0)
        todo &= ~ok
        scale *= 0.95  # an instance whose products grow starts nearer the origin
        if not bool(todo.any()):
            break
    mb = _Mpc()
    mb.T, mb.A, mb.B, mb.Q, mb.R, mb.x0 = (t.cpu().numpy() for t in (T, A, B, Q, R, x0))
    mb.u_max, mb.x_max = 1.0, 5.0
    return mb


# ---- what is measured ---------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "mpc":
        return {"kind": kind, "mpc": gb.BatchedMPC(_mpc_data(case, seed))}
    prec = PREC[case["prec"]]
    new = lambda count: torch.empty(count, dtype=torch.float64, device="cuda")
    if kind == "ipm":
        d = _ipm_data(case, seed)
        ctx = _context(case, tol=case["tol"])
        return {"kind": kind, "ctx": ctx, **d, "x": new(d["n"]), "s": new(d["mt"]), "lam": new(d["mt"])}
    if kind == "direction":
        d = _direction_data(case, seed)
        ctx = _context(case, formulation=FORM[case["form"]], ir_tol=1e-12)
        return {"kind": kind, "ctx": ctx, **d, "dx": new(d["n"]), "ds": new(d["mt"]), "dl": new(d["mt"])}
    d = _system_data(case, seed)
    # solutions to FP64 accuracy whatever the factor's arithmetic
    ctx = _context(case, ir_tol=1e-12)
    s = {"kind": kind, "ctx": ctx, "prec": prec, **d, "sol": torch.empty_like(d["rhs"])}
    if kind == "solve":
        ctx.kkt_assemble(d["val"], d["D"], REG, d["w"])
        ctx.kkt_factor(prec)
    return s


def run(s):
    kind = s["kind"]
    if kind == "mpc":
        m = s["mpc"]
        m.ipm_solve_batched(precision=gb.IPM_FP64, tol=1e-6)
        # (m.kkt, the residual left at the stopping point, is a difference of nearly equal numbers)
        return {"z": m.z, "objective": m.obj, "iterations": m.iters, "status": m.status}
    ctx = s["ctx"]
    if kind == "ipm":
        ctx.ipm_solve(s["val"], s["b"], s["c"], s["x"], s["s"], s["lam"], raise_on_error=True)
        return {"x": s["x"], "s": s["s"], "lam": s["lam"]}
    if kind == "direction":
        ctx.ipm_newton_direction(s["val"], s["b"], s["c"], s["x"], s["s"], s["lam"], s["target"],
                                 s["dx"], s["ds"], s["dl"])
        return {"dx": s["dx"], "ds": s["ds"], "dl": s["dl"]}
    if kind == "system":
        ctx.kkt_assemble(s["val"], s["D"], REG, s["w"])
        ctx.kkt_factor(s["prec"])
    ctx.kkt_solve(s["rhs"], s["sol"], gb.IPM_REFINE_PCG)
    return s["sol"]


# ---- the work that cannot be avoided ------------------------------------------
@functools.lru_cache(maxsize=64)
def _sizes(key):
    """nnz(J), nnz(K), nnz(L) and the factor's flops, from the symbolic analysis (host only)."""
    case = dict(key)
    n, m, rowptr, col, _, perm = _pattern(case)
    ctx = gb.IpmContext(n, m, rowptr, col, np.full(n, LOWER), np.full(n, UPPER),
                        options=gb.default_options(storage_fp64=0, formulation=FORM[case.get("form", "primal")]))
    i = ctx.kkt_analyze(_augmented_order(perm, m) if case.get("form") == "augmented" else perm)
    return int(rowptr[-1]), int(i.nnz_k), int(i.nnz_l), float(i.flops)


def work(case):
    """Every input read once and every output written once, J and D read once per product with
    K; the algorithmic flops of the factor (sum of colcount^2), the solves (two per entry of L
    and sweep) and, for whole solves, as many iterations as the problem class takes at least."""
    if case["kind"] == "mpc":
        stages = case["count"] * (case["t_min"] + case["t_max"]) / 2.0
        # ten iterations: K's blocks, a 16 x 16 block Cholesky and two solves per stage
        per_stage = 2.0 * (12 * 16 * 16 + 2 * 16 ** 3) + 2.0 * 4 * 16 * 16 * 2
        return {"bytes": 8.0 * stages * (144 + 48 + 16), "flops": 10.0 * stages * per_stage}
    nnz_j, nnz_k, nnz_l, flops = _sizes(tuple(sorted((k, v) for k, v in case.items() if k in
                                                     ("family", "x", "y", "z", "n", "m", "form"))))
    n, m = _pattern(case)[:2]
    mt = m + 2 * n
    word = 8.0 if PREC[case["prec"]] == gb.IPM_FP64 else 4.0
    one_solve = 2 * word * nnz_l + 8.0 * (nnz_j + mt + 2 * n)
    if case["kind"] == "solve":
        return {"bytes": case["nrhs"] * one_solve, "flops": 4.0 * nnz_l * case["nrhs"]}
    system = 8.0 * (nnz_j + mt + nnz_k) + word * nnz_l + one_solve
    if case["kind"] == "ipm":
        its = 8
        return {"bytes": its * (system + one_solve), "flops": its * (flops + 8.0 * nnz_l)}
    return {"bytes": system, "flops": flops + 4.0 * nnz_l}


# ---- the same results in plain 64-bit torch ------------------------------------
def _cg(apply, diag, b):
    """K x = b to the last bits: conjugate gradients with the diagonal as preconditioner,
    restarted on the true residual until it no longer falls."""
    x, best = torch.zeros_like(b), math.inf
    for _ in range(6):
        r = b - apply(x)
        now = float(r.norm())
        if now == 0.0 or now > 0.3 * best:
            break
        best = now
        dx, z = torch.zeros_like(b), r / diag
        p, rz = z.clone(), torch.dot(r, z)
        for k in range(6000):
            q = apply(p)
            a = rz / torch.dot(p, q)
            dx += a * p
            r = r - a * q
            if k % 16 == 15 and float(r.norm()) <= 1e-12 * now:
                break
            z = r / diag
            rz, old = torch.dot(r, z), rz
            p = z + (rz / old) * p
        x = x + dx
    return x


def _condensed(case, d, D):
    """K = W + J^T D J + D_l + D_u + delta_p as a product, and its diagonal."""
    n, m, rowptr, col, _, _ = _pattern(case)
    J = _Sparse(n, m, rowptr, col, d["val"])
    own = D[m:m + n] + D[m + n:] + REG
    if d["w"] is not None:
        own = own + d["w"]
    J2 = _Sparse(n, m, rowptr, col, d["val"] ** 2)
    return J, (lambda v: J.tmul(D[:m] * J.mul(v)) + own * v), J2.tmul(D[:m]) + own


def exact(case, seed):
    if case["kind"] == "mpc":
        return _exact_mpc(case, seed)
    if case["kind"] == "ipm":
        return _exact_ipm(case, seed)
    if case["kind"] == "direction":
        d = _direction_data(case, seed)
        m = d["m"]
        s, lam, x = d["s"], d["lam"], d["x"]
        D = 1.0 / (REG + s / lam)
        J, K, diag = _condensed(case, d, D)
        full = lambda v: torch.cat([J.mul(v), v, -v])
        n = d["n"]
        full_t = lambda v: J.tmul(v[:m]) + v[m:m + n] - v[m + n:]
        g = full(x) - torch.cat([d["b"], torch.full_like(x, LOWER), torch.full_like(x, -UPPER)])
        wl = d["target"] / lam
        dx = _cg(K, diag, -(d["c"] + full_t(D * (g - wl) - lam)))
        dl = D * (wl - g - full(dx))
        return {"dx": dx, "ds": -s + wl - (s / lam) * dl, "dl": dl}
    d = _system_data(case, seed)
    _, K, diag = _condensed(case, d, d["D"])
    return torch.stack([_cg(K, diag, b) for b in d["rhs"]])


def _exact_ipm(case, seed):
    """The LP's solution: a dense predictor-corrector method in 64 bits, run to the end."""
    d = _ipm_data(case, seed)
    n, m, rowptr, col, _, _ = _pattern(case)
    J = torch.zeros(m, n, dtype=torch.float64, device="cuda")
    J[torch.as_tensor(np.repeat(np.arange(m), np.diff(rowptr)), device="cuda"),
      torch.as_tensor(col, device="cuda").long()] = d["val"]
    full = lambda v: torch.cat([J @ v, v, -v])
    full_t = lambda v: J.t() @ v[:m] + v[m:m + n] - v[m + n:]
    x = torch.full((n,), 0.5 * (LOWER + UPPER), dtype=torch.float64, device="cuda")
    h = torch.cat([d["b"], torch.full_like(x, LOWER), torch.full_like(x, -UPPER)])
    s = torch.clamp(full(x) - h, min=1.0)
    lam = torch.ones_like(s)
    for _ in range(60):
        rp, rd = full(x) - h - s, d["c"] - full_t(lam)
        mu = torch.dot(s, lam) / len(s)
        if max(float(rp.abs().max()), float(rd.abs().max()), float(mu)) < 1e-11:
            break
        D = lam / s
        K = J.t() @ (D[:m, None] * J)
        K.diagonal().add_(D[m:m + n] + D[m + n:] + 1e-13)
        C, info = torch.linalg.cholesky_ex(K)
        if int(info):
            break

        def step(rc):  # s ds-target: lam ds + s dl = -rc
            rhs = -(rd - full_t(D * (-rp) - rc / s))
            dx = torch.cholesky_solve(rhs[:, None], C)[:, 0]
            ds = full(dx) + rp
            return dx, ds, (-rc - lam * ds) / s

        def most(v, dv):
            t = torch.where(dv < 0, -v / dv, torch.full_like(v, math.inf)).min()
            return torch.clamp(t, max=1.0)

        dx, ds, dl = step(s * lam)
        aff = torch.dot(s + most(s, ds) * ds, lam + most(lam, dl) * dl) / len(s)
        dx, ds, dl = step(s * lam + ds * dl - (aff / mu) ** 3 * mu)
        ap, ad = 0.995 * most(s, ds), 0.995 * most(lam, dl)
        x, s, lam = x + ap * dx, s + ap * ds, lam + ad * dl
    return {"x": x, "s": s, "lam": lam}


def _exact_mpc(case, seed):
    """The QPs' solutions: a primal-dual barrier method on the bounds that keeps the dynamics
    exact (it starts at u = 0, inside the box by construction); each step is one Riccati
    recursion over the stages, for all instances at once."""
    mb = _mpc_data(case, seed)
    dev = lambda a: torch.as_tensor(a, device="cuda")
    T, A, B, Q, R, x0 = (dev(a) for a in (mb.T, mb.A, mb.B, mb.Q, mb.R, mb.x0))
    count, top = len(T), int(T.max())
    off = torch.cumsum(T, 0) - T
    on = torch.arange(top, device="cuda")[None, :] < T[:, None]  # (count, top)
    at = torch.where(on, off[:, None] + torch.arange(top, device="cuda"), 0)
    A, B = A[at] * on[:, :, None, None], B[at] * on[:, :, None, None]
    W = torch.cat([R, Q], 1)[:, None, :].expand(count, top, 16)
    lim = torch.tensor([mb.u_max] * 4 + [mb.x_max] * 12, dtype=torch.float64, device="cuda")
    z = torch.zeros(count, top, 16, dtype=torch.float64, device="cuda")  # (u_k, x_{k+1})
    x = x0
    for k in range(top):
        x = (A[:, k] @ x[:, :, None])[:, :, 0]
        z[:, k, 4:] = x
    mask = on[:, :, None].to(torch.float64)
    lo, hi = torch.ones_like(z), torch.ones_like(z)  # multipliers of z + lim >= 0, lim - z >= 0
    for _ in range(80):
        sl, sh = z + lim, lim - z
        mu = ((lo * sl + hi * sh) * mask).sum((1, 2)) / (32.0 * T)
        if float(mu.max()) < 1e-13:
            break
        H = W + lo / sl + hi / sh
        t = (0.1 * mu)[:, None, None]
        q = W * z - t / sl + t / sh  # gradient of the barrier problem
        P = torch.zeros(count, 12, 12, dtype=torch.float64, device="cuda")
        p = torch.zeros(count, 12, dtype=torch.float64, device="cuda")
        gain, open_ = [None] * top, [None] * top
        for k in range(top - 1, -1, -1):
            act = on[:, k]
            S = torch.diag_embed(H[:, k, 4:]) + P
            v = q[:, k, 4:] + p
            BtS = B[:, k].transpose(1, 2) @ S
            M = torch.diag_embed(H[:, k, :4]) + BtS @ B[:, k]
            C = torch.linalg.cholesky(M)
            gain[k] = torch.cholesky_solve(BtS @ A[:, k], C)
            open_[k] = torch.cholesky_solve((q[:, k, :4] + (B[:, k].transpose(1, 2) @ v[:, :, None])[:, :, 0])[:, :, None], C)[:, :, 0]
            AtS = A[:, k].transpose(1, 2) @ S
            newP = AtS @ (A[:, k] - B[:, k] @ gain[k])
            newp = (A[:, k].transpose(1, 2) @ (v - (S @ (B[:, k] @ open_[k][:, :, None]))[:, :, 0])[:, :, None])[:, :, 0]
            P = torch.where(act[:, None, None], 0.5 * (newP + newP.transpose(1, 2)), P * 0)
            p = torch.where(act[:, None], newp, p * 0)
        dz = torch.zeros_like(z)
        dx = torch.zeros_like(x0)
        for k in range(top):
            du = -((gain[k] @ dx[:, :, None])[:, :, 0] + open_[k])
            dx = ((A[:, k] @ dx[:, :, None]) + (B[:, k] @ du[:, :, None]))[:, :, 0]
            dz[:, k, :4], dz[:, k, 4:] = du, dx
        dz = dz * mask
        dlo = t / sl - lo - lo / sl * dz
        dhi = t / sh - hi + hi / sh * dz

        def most(v, dv):
            r = torch.where((dv < 0) & on[:, :, None], -v / dv, torch.full_like(v, math.inf))
            return torch.clamp(0.995 * r.amin((1, 2)), max=1.0)

        ap = torch.minimum(most(sl, dz), most(sh, -dz))[:, None, None]
        ad = torch.minimum(most(lo, dlo), most(hi, dhi))[:, None, None]
        z, lo, hi = z + ap * dz, lo + ad * dlo, hi + ad * dhi
    obj = 0.5 * (W * z * z * mask).sum((1, 2))
    return {"z": z[on].reshape(-1), "objective": obj, "iterations": None, "status": None}
