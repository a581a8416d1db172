"""Performance cases of the sketched-FGMRES solver, each one call of a public entry point (or one forward and backward).

``listed()`` names the cases, ``draw(rng)`` gives another one of the same ranges, ``prepare`` makes what a program
holds before the call (matrix, right-hand side, solver handle), ``run`` is the call, ``work`` the bytes and operations
it cannot do without, and ``exact`` the same result from plain torch arithmetic in 64 bits.

The matrices are the package's own kinds: upwind convection-diffusion on a square or cubic grid (``convdiff``), a
random matrix with Zipf row lengths (``zipf``), and a batch of square grids (``batch``); all are made on the GPU.
"""
from __future__ import annotations

import math

import torch

from paper_2506_18408_gb300 import Solver, sfgmres_sketch_apply_noalloc, sfgmres_solve_autograd

SKETCH_SEED = 1
DEV = "cuda"


def listed():
    return [
        # the smallest solve in use: a 2D grid of 4,096 unknowns, one launch chain bound by latency
        {"name": "solve_2d_small", "kind": "solve", "matrix": "convdiff", "dim": 2, "side": 64, "beta": 20.0, "m": 30,
         "t": 2, "s": 120, "zeta": 8, "precision": "fp64", "tol": 1e-8, "max_outer": 20, "precond": False,
         "transpose": False},
        # the headline solve: a 3D grid of 2.1M unknowns in plain FP64
        {"name": "solve_3d", "kind": "solve", "matrix": "convdiff", "dim": 3, "side": 128, "beta": 50.0, "m": 100, "t": 2,
         "s": 400, "zeta": 8, "precision": "fp64", "tol": 1e-8, "max_outer": 50, "precond": False, "transpose": False},
        # the same system with FP32 inner cycles, for a user who wants more digits than the inner precision holds
        {"name": "solve_3d_fp32", "kind": "solve", "matrix": "convdiff", "dim": 3, "side": 128, "beta": 50.0, "m": 100,
         "t": 2, "s": 400, "zeta": 8, "precision": "fp32", "tol": 1e-12, "max_outer": 50, "precond": False,
         "transpose": False},
        # ILU(0) right preconditioning, a grid whose side is no power of two
        {"name": "solve_3d_ilu", "kind": "solve", "matrix": "convdiff", "dim": 3, "side": 96, "beta": 50.0, "m": 60, "t": 2,
         "s": 240, "zeta": 8, "precision": "fp64", "tol": 1e-8, "max_outer": 50, "precond": True, "transpose": False},
        # an unstructured matrix: rows of 4 to 256 entries at random columns, 50M entries
        {"name": "solve_zipf", "kind": "solve", "matrix": "zipf", "n": 2_000_000, "m": 60, "t": 4, "s": 240, "zeta": 8,
         "precision": "fp64", "tol": 1e-8, "max_outer": 50, "precond": False, "transpose": False},
        # many systems of uneven order with several right-hand sides each, solved together with FP32 inner cycles
        {"name": "batch_2d_fp32", "kind": "batch", "systems": 24, "lo": 32, "hi": 320, "nrhs": 4, "m": 40, "t": 2, "s": 160,
         "zeta": 8, "precision": "fp32", "tol": 1e-12, "max_outer": 60},
        # differentiation: 16 right-hand sides forward, the adjoint solves backward, gradients in b and in the values
        {"name": "grad_3d", "kind": "grad", "matrix": "convdiff", "dim": 3, "side": 64, "beta": 50.0, "nrhs": 16, "m": 50,
         "t": 2, "s": 200, "zeta": 8, "precision": "fp64", "tol": 1e-8, "max_outer": 50},
        # one preconditioner application (an inner cycle) for a program with its own outer iteration; an odd grid
        {"name": "cycle_3d_odd", "kind": "cycle", "matrix": "convdiff", "dim": 3, "side": 101, "beta": 30.0, "m": 60, "t": 3,
         "s": 240, "zeta": 8, "precision": "fp64"},
        # the same call with the paper's sketch: Clarkson-Woodruff (one nonzero per column), s = 1000, long cycles
        {"name": "cycle_3d_cw", "kind": "cycle", "matrix": "convdiff", "dim": 3, "side": 80, "beta": 50.0, "m": 200, "t": 2,
         "s": 1000, "zeta": 1, "precision": "fp64"},
        # y = A x, for a program's own residuals
        {"name": "spmv_3d", "kind": "spmv", "matrix": "convdiff", "dim": 3, "side": 128, "beta": 50.0},
        # c = S v through a handle
        {"name": "sketch", "kind": "sketch", "n": 2_097_152, "s": 400, "zeta": 8},
        # c = S v without a handle or any allocation, a ragged length
        {"name": "sketch_noalloc", "kind": "noalloc", "n": 1_000_003, "s": 240, "zeta": 8},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "batch", "grad", "cycle", "cycle", "spmv", "sketch", "noalloc"])
    if kind in ("sketch", "noalloc"):
        return {"kind": kind, "n": _log(rng, 5_000, 2_097_152), "s": rng.randint(100, 1000), "zeta": rng.choice([1, 4, 8])}
    if kind == "batch":
        lo = rng.randint(16, 64)
        return {"kind": "batch", "systems": rng.randint(3, 24), "lo": lo, "hi": lo + rng.randint(1, 200),
                "nrhs": rng.randint(1, 4), "m": 40, "t": rng.choice([2, 3]), "s": 160, "zeta": 8,
                "precision": rng.choice(["fp64", "fp32"]), "tol": 1e-12, "max_outer": 60}
    matrix = rng.choice(["convdiff", "convdiff", "convdiff", "zipf"])
    c = {"kind": kind, "matrix": matrix}
    if kind == "grad":
        matrix = c["matrix"] = "convdiff"
    if matrix == "zipf":
        c["n"] = _log(rng, 20_000, 1_500_000)
        size, t = c["n"] / 4, rng.choice([2, 4])
    else:
        c["dim"] = rng.choice([2, 3, 3])
        if c["dim"] == 3:
            c["side"] = _log(rng, 16, 64 if kind == "grad" else 128)
        else:
            c["side"] = _log(rng, 32, 160)
        c["beta"] = float(rng.randint(15, 50))
        size, t = c["side"] ** c["dim"], rng.choice([2, 2, 3])
    if kind == "spmv":
        return c
    c["m"] = rng.randint(30, 100) if size > 100_000 else rng.randint(20, 60)
    c["t"], c["s"], c["zeta"] = t, 4 * c["m"], 8
    c["precision"] = "fp64" if kind == "cycle" else rng.choice(["fp64", "fp64", "fp32"])
    if kind == "cycle":
        return c
    c["tol"] = 1e-8 if c["precision"] == "fp64" else 1e-12
    c["max_outer"] = 50
    if kind == "grad":
        c["nrhs"] = rng.randint(2, 16)
    else:
        c["transpose"] = rng.random() < 0.2
        c["precond"] = c["precision"] == "fp64" and matrix == "convdiff" and not c["transpose"] and rng.random() < 0.25
    return c


# ---- inputs ----------------------------------------------------------------------------------------------------------
def _gen(seed, stream):
    return torch.Generator(device=DEV).manual_seed(1_000_003 * int(seed) + stream)


def _convdiff(dim, side, beta):
    """Upwind finite differences of -Laplace(u) + beta . grad(u), rows scaled by h^2, x fastest, columns increasing."""
    n, h = side ** dim, 1.0 / (side + 1)
    idx = torch.arange(n, device=DEV)
    offs, vals, keep = [], [], []
    for c in reversed(range(dim)):
        offs.append(-(side ** c))
        vals.append(-1.0 - h * beta[c])
        keep.append((idx // side ** c) % side > 0)
    offs.append(0)
    vals.append(2.0 * dim + h * sum(beta[:dim]))
    keep.append(torch.ones(n, dtype=torch.bool, device=DEV))
    for c in range(dim):
        offs.append(side ** c)
        vals.append(-1.0)
        keep.append((idx // side ** c) % side < side - 1)
    keep = torch.stack(keep, 1)
    col = idx[:, None] + torch.tensor(offs, device=DEV)
    val = torch.tensor(vals, dtype=torch.float64, device=DEV).expand(n, -1)
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(keep.sum(1), 0, out=rp[1:])
    return rp, col[keep].to(torch.int32), val[keep]


def _zipf(n, seed):
    """Row lengths Zipf(1.5) clipped to [4, 256], uniform columns, N(0,1) values, diagonal 1.2 x the absolute row sum."""
    g = _gen(seed, 0)
    p = torch.arange(1, 257, dtype=torch.float64) ** -1.5
    p[255] += 2.612375348685488 - float(p.sum())  # zeta(1.5): the tail beyond 256
    p[3] += p[:3].sum()
    p[:3] = 0.0
    cdf = torch.cumsum(p, 0).to(DEV) / p.sum().item()
    length = (torch.searchsorted(cdf, torch.rand(n, generator=g, device=DEV, dtype=torch.float64)) + 1).clamp_(4, min(256, n))
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), length - 1)
    key = rows * n + torch.randint(0, n, rows.shape, generator=g, device=DEV)
    key = torch.unique(torch.cat([key, torch.arange(n, device=DEV) * (n + 1)]))  # sorted, the diagonal among them
    rows, col = key // n, key % n
    # multiples of 2^-20, so that the sums below are exact and the matrix is the same each time
    val = torch.round(torch.randn(key.shape, generator=g, device=DEV, dtype=torch.float64) * 2.0**20) / 2.0**20
    diag = rows == col
    val[diag] = 0.0
    rp = torch.searchsorted(rows, torch.arange(n + 1, device=DEV))
    total = torch.cat([torch.zeros(1, device=DEV, dtype=torch.float64), torch.cumsum(val.abs(), 0)])
    val[diag] = 1.2 * (total[rp[1:]] - total[rp[:-1]])
    return rp, col.to(torch.int32), val


def _batch(case, seed):
    """Square grids with sides U{lo..hi} and beta ~ U(0,50)^2 per system as one block-diagonal matrix.  The sides follow
    from the case alone, so that every seed is the same amount of work."""
    g = torch.Generator().manual_seed(case["systems"] * 1000 + case["hi"])
    sides = torch.randint(case["lo"], case["hi"] + 1, (case["systems"],), generator=g).tolist()
    beta = (50.0 * torch.rand(case["systems"], 2, generator=g, dtype=torch.float64)).tolist()
    rps, cols, vals, n, nnz = [torch.zeros(1, dtype=torch.int64, device=DEV)], [], [], 0, 0
    for q, side in enumerate(sides):
        rp, col, val = _convdiff(2, side, beta[q])
        rps.append(rp[1:] + nnz)
        cols.append(col + n)
        vals.append(val)
        n, nnz = n + side * side, nnz + val.numel()
    return [side * side for side in sides], torch.cat(rps), torch.cat(cols), torch.cat(vals)


def _beta(case):
    return [case["beta"], 0.6 * case["beta"], 0.2 * case["beta"]] if case["dim"] == 3 else [case["beta"], 0.5 * case["beta"]]


def _matrix(case, seed):
    """(orders, row pointers, columns, values)."""
    if case["kind"] == "batch":
        return _batch(case, seed)
    if case["kind"] == "sketch":  # the handle's matrix plays no part in S v: the identity
        n = case["n"]
        return n, torch.arange(n + 1, device=DEV), torch.arange(n, device=DEV, dtype=torch.int32), \
            torch.ones(n, device=DEV, dtype=torch.float64)
    if case["matrix"] == "zipf":
        return (case["n"], *_zipf(case["n"], seed))
    return (case["side"] ** case["dim"], *_convdiff(case["dim"], case["side"], _beta(case)))


def _order(case):
    return case["n"] if "n" in case else case["side"] ** case["dim"]


def _vector(case, seed, n, stream=1):
    if case.get("matrix") == "zipf":
        return 2.0 * torch.rand(n, generator=_gen(seed, stream), device=DEV, dtype=torch.float64) - 1.0
    return torch.randn(n, generator=_gen(seed, stream), device=DEV, dtype=torch.float64)


def _inputs(case, seed, n):
    """The dense inputs of a call: b (or v, x), and the target of the loss."""
    kind = case["kind"]
    if kind == "batch":
        return (_vector(case, seed, case["nrhs"] * n),)
    if kind == "grad":
        return (_vector(case, seed, case["nrhs"] * n).view(case["nrhs"], n),
                _vector(case, seed, case["nrhs"] * n, 2).view(case["nrhs"], n))
    v = _vector(case, seed, n)
    return (v / v.norm() if kind == "cycle" else v,)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "noalloc":
        v = _vector(case, seed, case["n"])
        return {"case": case, "in": (v,), "c": torch.empty(case["s"], dtype=torch.float64, device=DEV)}
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        n, rp, col, val = _matrix(case, seed)
        opt = {k: case[k] for k in ("zeta", "precision", "max_outer") if k in case}
        if case.get("precond"):
            opt["precond"] = 1
        solver = Solver(n, rp, col, val, sketch_seed=SKETCH_SEED, **opt)
        state = {"case": case, "solver": solver, "stream": stream, "in": _inputs(case, seed, solver.n)}
        if kind == "grad":
            state["vals"] = val.clone().requires_grad_()
            state["b"] = state["in"][0].clone().requires_grad_()
    stream.synchronize()
    return state


# ---- the calls -------------------------------------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "noalloc":
        sfgmres_sketch_apply_noalloc(case["n"], case["s"], case["zeta"], SKETCH_SEED, state["in"][0], state["c"],
                                     torch.cuda.current_stream().cuda_stream)
        return state["c"]
    solver = state["solver"]
    with torch.cuda.stream(state["stream"]):
        if kind == "spmv":
            return solver.spmv(state["in"][0])
        if kind == "sketch":
            return solver.sketch(state["in"][0], case["s"])
        par = {"m": case["m"], "s": case["s"], "k": case["t"]}
        if kind == "cycle":
            z, k, _, _, _ = solver.inner_cycle(state["in"][0], basis=False, **par)
            return {"z": z, "k": k}
        if kind == "solve":
            return solver.solve(state["in"][0], tol=case["tol"], transpose=case["transpose"], **par)[0]
        if kind == "batch":
            return solver.solve_batch(state["in"][0], nrhs=case["nrhs"], tol=case["tol"], **par)[0]
        x = sfgmres_solve_autograd(solver, state["vals"], state["b"], tol=case["tol"], **par)
        loss = ((x - state["in"][1]) ** 2).sum()
        gb, gv = torch.autograd.grad(loss, (state["b"], state["vals"]))
        return {"x": x.detach(), "grad_b": gb, "grad_vals": gv}


# ---- what a call cannot do without -----------------------------------------------------------------------------------
def _shape(case):
    """(unknowns, stored entries) of the matrix, near enough for a count of bytes."""
    if case["kind"] == "batch":
        n = case["systems"] * (case["lo"] ** 2 + case["lo"] * case["hi"] + case["hi"] ** 2) / 3.0
        return n, 5 * n
    n = _order(case)
    if case["matrix"] == "zipf":
        return n, 25.4 * n
    return n, (2 * case["dim"] + 1) * n - 2 * case["dim"] * n / case["side"]


def _cycles(case):
    """Inner cycles of m steps that a solve of this kind takes, near enough for a count of bytes."""
    if case["matrix" if "matrix" in case else "kind"] == "zipf":
        return 16.0
    if case.get("precond"):
        return 3.0
    if case.get("dim") == 3:
        return max(1.0, 0.03 * case["side"]) * 100.0 / case["m"] * (1.5 if case["tol"] < 1e-9 else 1.0)
    side = case.get("side") or 0.5 * (case["lo"] + case["hi"])
    return max(1.0, 0.1 * side) * 40.0 / case["m"]


def work(case):
    kind = case["kind"]
    if kind in ("sketch", "noalloc"):
        return {"bytes": 8.0 * (case["n"] + case["s"]), "flops": 1.0 * case["n"] * case["zeta"]}
    n, nnz = _shape(case)
    if kind == "spmv":
        return {"bytes": 12.0 * nnz + 4.0 * n + 16.0 * n, "flops": 2.0 * nnz}
    m, t = case["m"], case["t"]
    w = 8 if case["precision"] == "fp64" else 4
    rhs = case.get("nrhs", 1)
    # an inner step: A once, u_i read, w' written and read, the window read, u_{i+1} written (S is hashed: no bytes)
    step = nnz * (w + 4) + 4 * n + rhs * (2 * t + 3) * n * w
    step_f = rhs * (2 * nnz + (4 * t + 2) * n + case["zeta"] * n)
    cycle = m * step + rhs * ((m + 1) * n * w + 8 * n)  # and z = B y
    cycle_f = m * step_f + rhs * 2 * m * n
    if kind == "cycle":
        return {"bytes": float(cycle), "flops": float(cycle_f)}
    cycles = _cycles(case) * (2 if kind == "grad" else 1)
    outer = 12 * nnz + rhs * 8 * n * (2 * cycles + 4)  # w = A z_j and two passes against v_0..v_j, on the mean
    return {"bytes": float(cycles * (cycle + outer)), "flops": float(cycles * (cycle_f + 2 * rhs * nnz))}


# ---- the same results in plain torch, 64 bits ------------------------------------------------------------------------
def _csr(rp, col, val, n):
    return torch.sparse_csr_tensor(rp, col.to(torch.int64), val, size=(n, n))


def _transposed(rp, col, val, n):
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1])
    order = torch.argsort(col.to(torch.int64) * n + rows)
    rpt = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(col.to(torch.int64), minlength=n), 0, out=rpt[1:])
    return rpt, rows[order], val[order]


def _bicgstab(A, R, dinv, cut, steps):
    """Approximate solutions of A X = R, columns independent, with diagonal preconditioning, to cut x the norm of R."""
    X = torch.zeros_like(R)
    r, r0 = R.clone(), R.clone()
    rho = alpha = om = torch.ones(R.shape[1], dtype=torch.float64, device=DEV)
    v = p = torch.zeros_like(R)
    goal = cut * R.norm(dim=0)
    best, left = X, r.norm(dim=0)
    for it in range(steps):
        rho1 = (r0 * r).sum(0)
        b = rho1 / rho * (alpha / om)
        p = r + b * (p - om * v)
        ph = dinv * p
        v = A @ ph
        alpha = rho1 / (r0 * v).sum(0)
        s = r - alpha * v
        sh = dinv * s
        t = A @ sh
        om = (t * s).sum(0) / (t * t).sum(0)
        X = X + alpha * ph + om * sh
        r = s - om * t
        rho = rho1
        now = r.norm(dim=0)
        live = torch.isfinite(now) & (now <= left)
        best, left = torch.where(live, X, best), torch.where(live, now, left)
        if it % 8 == 7 and (bool((left <= goal).all()) or not bool(torch.isfinite(now).any())):
            break
    return best


def _solve(rp, col, val, n, B):
    """A^{-1} B (B: n x nrhs) by refinement: corrections from BiCGSTAB until the residual stops falling."""
    A = _csr(rp, col, val, n)
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1])
    d = torch.zeros(n, dtype=torch.float64, device=DEV)
    d[rows[rows == col]] = val[rows == col]
    dinv = (1.0 / d)[:, None]
    X, R, last = torch.zeros_like(B), B, math.inf
    for _ in range(40):
        Y = X + _bicgstab(A, R, dinv, 1e-7, 600)
        S = B - A @ Y
        now = float((S.norm(dim=0) / B.norm(dim=0)).max())
        if not now < 0.7 * last:
            break
        X, R, last = Y, S, now
    return X


def _mix(z):
    """The output function of SplitMix64 on int64 values taken as unsigned."""
    z = (z ^ ((z >> 30) & ((1 << 34) - 1))) * (0xBF58476D1CE4E5B9 - (1 << 64))
    z = (z ^ ((z >> 27) & ((1 << 37) - 1))) * (0x94D049BB133111EB - (1 << 64))
    return z ^ ((z >> 31) & ((1 << 33) - 1))


def _sketch(n, s, zeta):
    """The embedding S as a sparse matrix (s x n): slot q = j zeta + l takes its row from outputs 128 q + 2 a of the
    counter form (the first not used by the column's earlier slots), its sign from output 128 q + 1."""
    gamma = 0x9E3779B97F4A7C15 - (1 << 64)

    def out(k):
        return _mix(SKETCH_SEED + (k + 1) * gamma)

    j = torch.arange(n, device=DEV)
    rows, signs = [], []
    for l in range(zeta):
        base = (j * zeta + l) * 128
        row = torch.full((n,), -1, device=DEV)
        todo = torch.ones(n, dtype=torch.bool, device=DEV)
        for a in range(64):
            cand = (((out(base + 2 * a) >> 32) & 0xFFFFFFFF) * s) >> 32
            row = torch.where(todo, cand, row)
            todo = torch.zeros(n, dtype=torch.bool, device=DEV)
            for r in rows:
                todo |= r == row
            if not bool(todo.any()):
                break
        rows.append(row)
        signs.append(torch.where(out(base + 1) < 0, -1.0, 1.0).to(torch.float64))
    rows, signs, cols = torch.cat(rows), torch.cat(signs), j.repeat(zeta)
    order = torch.argsort(rows * n + cols)
    rp = torch.zeros(s + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(rows, minlength=s), 0, out=rp[1:])
    return torch.sparse_csr_tensor(rp, cols[order], signs[order] / math.sqrt(zeta), size=(s, n))


def _cycle(case, A, v, n):
    """z = B y of one cycle: the truncated-Arnoldi basis B, y the least-squares solution of S A B y = S v."""
    S, m, t = _sketch(n, case["s"], case["zeta"]), case["m"], case["t"]
    B = torch.empty(m, n, dtype=torch.float64, device=DEV)
    C = torch.empty(case["s"], m, dtype=torch.float64, device=DEV)
    B[0] = v
    for i in range(m):
        w = A @ B[i]
        C[:, i] = S @ w
        if i + 1 < m:
            W = B[max(0, i - t + 1):i + 1]
            w = w - W.T @ (W @ w)
            B[i + 1] = w / w.norm()
    Q, R = torch.linalg.qr(C)
    y = torch.linalg.solve_triangular(R, (Q.T @ (S @ v))[:, None], upper=True)[:, 0]
    return B.T @ y


def exact(case, seed):
    kind = case["kind"]
    if kind in ("sketch", "noalloc"):
        return _sketch(case["n"], case["s"], case["zeta"]) @ _vector(case, seed, case["n"])
    n, rp, col, val = _matrix(case, seed)
    orders = n
    n = rp.numel() - 1
    given = _inputs(case, seed, n)
    if kind == "spmv":
        return _csr(rp, col, val, n) @ given[0]
    if kind == "cycle":
        return {"z": _cycle(case, _csr(rp, col, val, n), given[0], n), "k": None}
    if kind == "solve":
        if case["transpose"]:
            rp, col, val = _transposed(rp, col, val, n)
        return _solve(rp, col, val, n, given[0][:, None])[:, 0]
    nrhs = case["nrhs"]
    if kind == "batch":  # problem order (system by system, its right-hand sides in turn) to one column per right-hand side
        parts = given[0].split([nrhs * k for k in orders])
        X = _solve(rp, col, val, n, torch.cat([p.view(nrhs, k).T for p, k in zip(parts, orders)]))
        return torch.cat([p.T.reshape(-1) for p in X.split(list(orders))])
    X = _solve(rp, col, val, n, given[0].T.contiguous())
    L = _solve(*_transposed(rp, col, val, n), n, 2.0 * (X - given[1].T))
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1])
    gv = torch.zeros_like(val)
    for r in range(nrhs):
        gv -= L[rows, r] * X[col.to(torch.int64), r]
    return {"x": X.T.contiguous(), "grad_b": L.T.contiguous(), "grad_vals": gv}
