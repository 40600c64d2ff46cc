"""What the library is timed on: the work its users have it do, at the sizes they have.

Every case goes through the public entry points of `paper_2608_09647_gb300`.  The matrices
are the families of this repository's benchmark (5-/9-point and 7-point grids, 27-point
diffusion with uneven coefficients, rotated Q1 elements, power-law graphs), assembled here
with torch on the GPU.  Most carry a reaction term (`shift`, relative to the diagonal), as
an implicit time step has it.  Right-hand sides are b = A x* of a random x*, and solves go
to 1e-12, near the accuracy of a direct solver, so that x is settled to about 1e-10.
"""
import math
import os

import numpy as np
import torch

import paper_2608_09647_gb300 as cg

TOL = 1e-12
MAXIT = 20000
PRECOND = {"none": cg.CG_PRECOND_NONE, "jacobi": cg.CG_PRECOND_JACOBI, "fsai": cg.CG_PRECOND_FSAI}
PRECISION = {"fp64": cg.CG_PREC_FP64, "ir": cg.CG_PREC_FP32_IR, "ru": cg.CG_PREC_FP32_RU}


def listed():
    return [
        # a small system inside an outer loop (a Newton or time step): latency of one solve
        {"name": "cg_5pt_64", "do": "solve", "matrix": "grid2d", "side": 64, "points": 5, "eps": 1.0, "shift": 0.0,
         "precond": "none", "precision": "fp64"},
        # the same from a plugin that may not allocate device memory
        {"name": "noalloc_5pt_48", "do": "noalloc", "matrix": "grid2d", "side": 48, "points": 5, "eps": 0.5,
         "shift": 1e-3, "precond": "jacobi", "precision": "fp64"},
        # an ordinary 2-D problem: larger than a cluster's shared memory, far smaller than L2
        {"name": "jacobi_9pt_301", "do": "solve", "matrix": "grid2d", "side": 301, "points": 9, "eps": 0.05,
         "shift": 1e-3, "precond": "jacobi", "precision": "fp64"},
        # the headline size: a 3-D field of 16.8 M unknowns, memory-sized vectors
        {"name": "jacobi_7pt_256", "do": "solve", "matrix": "grid3d", "side": 256, "points": 7, "shift": 1e-3,
         "precond": "jacobi", "precision": "fp64"},
        # 3-D diffusion with uneven coefficients, fp32 with fp64 reliable updates
        {"name": "ru_27pt_160", "do": "solve", "matrix": "grid3d", "side": 160, "points": 27, "shift": 1e-3,
         "precond": "jacobi", "precision": "ru"},
        # a matrix without structure (a network): rows of 1 to a few hundred entries
        {"name": "jacobi_graph_2m", "do": "solve", "matrix": "graph", "n": 2000000, "precond": "jacobi",
         "precision": "fp64"},
        # one product with such a matrix, as an outside Krylov or eigenvalue code calls it
        {"name": "spmv_graph_3m", "do": "spmv", "matrix": "graph", "n": 3000001},
        # many independent systems of uneven size in one call
        {"name": "batch_96", "do": "batch", "count": 96, "side_lo": 32, "side_hi": 512, "shift": 1e-3,
         "precision": "fp64"},
        # fewer and smaller ones, fp32 with fp64 reliable updates
        {"name": "batch_ru_24", "do": "batch", "count": 24, "side_lo": 33, "side_hi": 200, "shift": 1e-3,
         "precision": "ru"},
        # learned FSAI preconditioner on rotated Q1 elements
        {"name": "fsai_ru_q1_1000", "do": "solve", "matrix": "q1", "side": 1000, "theta": 0.7, "eps": 0.01,
         "shift": 1e-3, "precond": "fsai", "precision": "ru"},
        # one gradient of the preconditioner's training, at its training sizes
        {"name": "fsai_train_q1_64", "do": "train", "matrix": "q1", "side": 64, "theta": 1.1, "eps": 0.03,
         "shift": 0.0},
        # a matrix that is new at every call (a coefficient that moves): set up, solve, give back
        {"name": "fresh_7pt_97", "do": "fresh", "matrix": "grid3d", "side": 97, "points": 7, "shift": 1e-2,
         "precond": "jacobi", "precision": "fp64"},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    shift = float("%.3g" % _log(rng, 1e-3, 2e-2))
    eps = float("%.3g" % _log(rng, 1e-2, 1.0))
    points = rng.choice([5, 9])
    kind = rng.choice(["small", "noalloc", "grid2d", "grid3d", "refine", "graph", "spmv", "batch", "fsai", "train",
                       "fresh", "fresh_fsai"])
    if kind in ("small", "noalloc", "grid2d"):
        lo, hi = {"small": (20, 128), "noalloc": (20, 128), "grid2d": (129, 1500)}[kind]
        pc = "jacobi" if kind == "noalloc" else rng.choice(["none", "jacobi"])
        return {"do": "noalloc" if kind == "noalloc" else "solve", "matrix": "grid2d", "side": round(_log(rng, lo, hi)),
                "points": points, "eps": eps, "shift": shift, "precond": pc, "precision": "fp64"}
    if kind == "grid3d":
        return {"do": "solve", "matrix": "grid3d", "side": round(_log(rng, 26, 250)), "points": 7, "shift": shift,
                "precond": rng.choice(["none", "jacobi"]), "precision": "fp64"}
    if kind == "refine":
        return {"do": "solve", "matrix": "grid3d", "side": round(_log(rng, 24, 155)), "points": rng.choice([7, 27, 27]),
                "shift": shift, "precond": "jacobi", "precision": rng.choice(["ru", "ru", "ir"])}
    if kind == "graph":
        return {"do": "solve", "matrix": "graph", "n": round(_log(rng, 2e4, 2e6)), "precond": "jacobi",
                "precision": rng.choice(["fp64", "fp64", "ru"])}
    if kind == "spmv":
        if rng.random() < 0.7:
            return {"do": "spmv", "matrix": "graph", "n": round(_log(rng, 2e4, 3e6))}
        return {"do": "spmv", "matrix": "grid3d", "side": round(_log(rng, 24, 160)), "points": rng.choice([7, 27]),
                "shift": shift}
    if kind == "batch":
        lo = round(_log(rng, 12, 64))
        return {"do": "batch", "count": round(_log(rng, 8, 96)), "side_lo": lo, "side_hi": round(_log(rng, lo + 16, 400)),
                "shift": shift, "precision": rng.choice(["fp64", "ru"])}
    if kind == "train":
        return {"do": "train", "matrix": "q1", "side": round(_log(rng, 24, 160)), "theta": round(rng.uniform(0.0, 3.1), 2),
                "eps": eps, "shift": 0.0}
    if kind == "fresh":
        return {"do": "fresh", "matrix": "grid3d", "side": round(_log(rng, 20, 128)), "points": 7, "shift": shift,
                "precond": "jacobi", "precision": "fp64"}
    return {"do": "solve" if kind == "fsai" else "fresh", "matrix": "q1", "side": round(_log(rng, 100, 900)),
            "theta": round(rng.uniform(0.0, 3.1), 2), "eps": eps, "shift": shift, "precond": "fsai", "precision": "ru"}


# ---------------------------------------------------------------- matrices

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _compress(n, deltas, vals, mask):
    """CSR (int32, int32, float64) of an [n, K] table whose column k lies at i + deltas[k], deltas ascending."""
    rows = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rows[1:] = torch.cumsum(mask.sum(1), 0)
    i = torch.arange(n, dtype=torch.int32, device="cuda")
    cols = i[:, None] + torch.tensor(deltas, dtype=torch.int32, device="cuda")
    return rows.to(torch.int32), cols[mask], vals[mask]


def _product(deltas, vals, mask, x):
    """A x for the same table."""
    i = torch.arange(x.numel(), dtype=torch.int64, device="cuda")
    y = torch.zeros_like(x)
    for k, d in enumerate(deltas):
        y += torch.where(mask[:, k], vals[:, k] * x[(i + d).clamp_(0, x.numel() - 1)], 0.0)
    return y


def _grid(side, offsets, weight, shift):
    """Graph Laplacian table of a Dirichlet grid: -weight(o) towards each offset o = (dz, dy, dx), the sum of all
    weights (neighbours outside included) times 1 + shift on the diagonal."""
    dim = 3 if any(o[0] for o in offsets) else 2
    zs = side if dim == 3 else 1
    n = zs * side * side
    i = torch.arange(n, device="cuda")
    z, y, x = i // (side * side), (i // side) % side, i % side
    offsets = sorted(offsets + [(0, 0, 0)])
    deltas = [(o[0] * side + o[1]) * side + o[2] for o in offsets]
    vals = torch.empty((n, len(offsets)), dtype=torch.float64, device="cuda")
    mask = torch.empty((n, len(offsets)), dtype=torch.bool, device="cuda")
    diag = torch.zeros(n, dtype=torch.float64, device="cuda")
    for k, o in enumerate(offsets):
        zz, yy, xx = z + o[0], y + o[1], x + o[2]
        mask[:, k] = (zz >= 0) & (zz < zs) & (yy >= 0) & (yy < side) & (xx >= 0) & (xx < side)
        if o != (0, 0, 0):
            w = weight(o, (z, y, x), (zz, yy, xx))
            vals[:, k] = -w
            diag += w
    vals[:, offsets.index((0, 0, 0))] = diag * (1.0 + shift)
    return deltas, vals, mask


def _grid2d(side, points, eps, shift):
    offsets = [(0, a, b) for a in (-1, 0, 1) for b in (-1, 0, 1) if (a or b) and (points == 9 or not (a and b))]

    def weight(o, u, v):
        return (1.0 + eps) / 4 if o[1] and o[2] else eps if o[2] else 1.0
    return _grid(side, offsets, weight, shift)


def _grid3d(side, points, shift, gen):
    """7-point: unit couplings.  27-point: couplings sqrt(c_u c_v) of a lognormal coefficient c at every node."""
    every = [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1) if a or b or c]
    if points == 7:
        return _grid(side, [o for o in every if sum(map(abs, o)) == 1], lambda o, u, v: 1.0, shift)
    m = side + 2
    c = torch.exp(torch.randn((m * m * m,), dtype=torch.float64, device="cuda", generator=gen))

    def weight(o, u, v):
        at = [((p[0] + 1) * m + p[1] + 1) * m + p[2] + 1 for p in (u, v)]
        return torch.sqrt(c[at[0]] * c[at[1]]) * 0.5 ** (sum(map(abs, o)) - 1)
    return _grid(side, every, weight, shift)


def _q1(side, theta, eps, shift, gen):
    """Q1 stiffness of a_c R diag(1, eps) R^T with lognormal a_c per cell (exact element matrices)."""
    c, s = math.cos(theta), math.sin(theta)
    kxx, kyy, kxy = c * c + eps * s * s, s * s + eps * c * c, (1.0 - eps) * c * s
    sg, M = (-1.0, 1.0), ((1 / 3, 1 / 6), (1 / 6, 1 / 3))
    a = torch.exp(1.5 * torch.randn((side + 1, side + 1), dtype=torch.float64, device="cuda", generator=gen))
    n = side * side
    offsets = [(dy, dx) for dy in (-1, 0, 1) for dx in (-1, 0, 1)]
    vals = torch.zeros((n, 9), dtype=torch.float64, device="cuda")
    mask = torch.empty((n, 9), dtype=torch.bool, device="cuda")
    i = torch.arange(n, device="cuda")
    y, x = i // side, i % side
    for k, (dy, dx) in enumerate(offsets):
        v = torch.zeros((side, side), dtype=torch.float64, device="cuda")
        for cy in (0, 1):  # the cells around a node: local node (1 - cx, 1 - cy) of cell (x + cx, y + cy)
            for cx in (0, 1):
                p, q = 1 - cx, 1 - cy
                r, t = p + dx, q + dy
                if 0 <= r <= 1 and 0 <= t <= 1:
                    ke = kxx * sg[p] * sg[r] * M[q][t] + kyy * sg[q] * sg[t] * M[p][r] \
                        + kxy * (sg[p] * sg[t] + sg[q] * sg[r]) / 4
                    v += a[cy:cy + side, cx:cx + side] * ke
        vals[:, k] = v.reshape(-1) * (1.0 + shift if (dy, dx) == (0, 0) else 1.0)
        mask[:, k] = (x + dx >= 0) & (x + dx < side) & (y + dy >= 0) & (y + dy < side)
    return [dy * side + dx for dy, dx in offsets], vals, mask


def _graph(n, gen):
    """Weighted graph Laplacian with power-law degrees, 70 % of the couplings within 64 rows, the others anywhere."""
    def rand(k):
        return torch.rand(k, dtype=torch.float64, device="cuda", generator=gen)
    half = ((2.0 * rand(n).clamp_min(1e-12).pow(-1.0 / 1.6)).floor().clamp(max=600.0) + 1.0).div(2.0).floor().long()
    i = torch.repeat_interleave(torch.arange(n, device="cuda"), half)
    near = rand(i.numel()) < 0.7
    u = rand(i.numel())
    j = torch.where(near, i + ((2.0 * u - 1.0) * 64.5).floor().long(), (u * n).floor().long())
    w = 0.5 + rand(i.numel())
    keep = (j >= 0) & (j < n) & (j != i)
    i, j, w = i[keep], j[keep], w[keep]
    key, order = torch.sort(torch.minimum(i, j) * n + torch.maximum(i, j), stable=True)
    key, count = torch.unique_consecutive(key, return_counts=True)  # an edge drawn twice weighs both
    w = torch.segment_reduce(w[order], "sum", lengths=count)
    i, j = key // n, key % n
    key, order = torch.sort(torch.cat([key, j * n + i, torch.arange(n, device="cuda") * (n + 1)]))
    val = torch.cat([w, w, torch.zeros(n, dtype=torch.float64, device="cuda")])[order]
    row, col = key // n, key % n
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    total = torch.segment_reduce(val, "sum", offsets=rowptr)
    scale = 1.0 + 10.0 ** (rand(n) - 2.5)
    on = row == col
    val = torch.where(on, torch.where(total > 0, scale * total, 1.0)[row], -val)
    return rowptr.to(torch.int32), col.to(torch.int32), val


def _matrix(case, gen, x):
    """CSR of the case's matrix and its product with x (or the table, for x None)."""
    if case["matrix"] == "graph":
        rowptr, col, val = _graph(case["n"], gen)
        return (rowptr, col, val), torch.segment_reduce(val * x[col.long()], "sum", offsets=rowptr.long())
    if case["matrix"] == "grid2d":
        table = _grid2d(case["side"], case["points"], case["eps"], case["shift"])
    elif case["matrix"] == "grid3d":
        table = _grid3d(case["side"], case["points"], case["shift"], gen)
    else:
        table = _q1(case["side"], case["theta"], case["eps"], case["shift"], gen)
    csr = _compress(table[1].shape[0], *table)
    return csr, table if x is None else _product(*table, x)


def _rows(case):
    return case["n"] if case["matrix"] == "graph" else case["side"] ** (3 if case["matrix"] == "grid3d" else 2)


def _xstar(n, gen):
    return 2.0 * torch.rand(n, dtype=torch.float64, device="cuda", generator=gen) - 1.0


def _members(case, seed):
    """(side, points, eps) of a batch: uneven sides, 5- and 9-point in turn, eps over three decades.  The sizes belong
    to the case, the coefficients to the seed."""
    sizes = np.random.RandomState(case["count"] * 1009 + case["side_lo"])
    values = np.random.RandomState(seed % (1 << 31))
    return [(int(sizes.randint(case["side_lo"], case["side_hi"] + 1)), 5 if k % 2 == 0 else 9,
             float(10.0 ** (-3.0 * values.random_sample()))) for k in range(case["count"])]


def _weights():
    w = np.load(os.path.join(os.path.dirname(cg.__file__), "fsai_q1aniso_bf16.npy"))
    return (w.astype(np.uint32) << 16).view(np.float32)


# ---------------------------------------------------------------- the passes

def _check(status, h=None):
    if status != cg.CG_OK:
        raise RuntimeError("status %d: %s" % (status, cg.cg_last_error(h)))


def prepare(case, seed):
    gen = _generator(seed)
    s = {"case": case}
    if case["do"] == "batch":
        systems, xs = [], []
        for side, points, eps in _members(case, seed):
            table = _grid2d(side, points, eps, case["shift"])
            xs.append(_xstar(side * side, gen))
            systems.append((_compress(side * side, *table), _product(*table, xs[-1])))
        # one buffer for all right-hand sides and one for all solutions, systems on 16-byte boundaries
        starts = np.concatenate([[0], np.cumsum([(x.numel() + 1) // 2 * 2 for x in xs])])
        s["starts"] = [(int(a), x.numel()) for a, x in zip(starts, xs)]
        s["total"] = int(starts[-1])
        b = torch.zeros(s["total"], dtype=torch.float64, device="cuda")
        for (a, n), (_, v) in zip(s["starts"], systems):
            b[a:a + n] = v
        s["b"] = b
        s["h"] = cg.cg_batch_create([m[0][0] for m in systems], [m[0][1] for m in systems], [m[0][2] for m in systems])
        _batch(s, 1)  # the handle's schedule is chosen at its first solve
        return s
    n = _rows(case)
    if case["do"] == "train":
        s["csr"], s["table"] = _matrix(case, gen, None)
        deltas, vals, mask = s["table"]
        d = vals[:, 4]
        x, b, snaps = torch.zeros_like(d), _product(*s["table"], _xstar(n, gen)), []
        for k in range(1, 33):  # residuals of a relaxation after 2, 8 and 32 sweeps
            r = b - _product(*s["table"], x)
            x += 0.6 * r / d
            if k in (2, 8, 32):
                snaps.append(b - _product(*s["table"], x))
        s["resid"] = torch.stack(snaps)
        noise = torch.randn(cg.CG_MLP_PARAMS, device="cuda", generator=gen)
        s["params"] = torch.from_numpy(_weights().copy()).cuda() * (1.0 + 0.05 * noise)
        s["h"] = cg.cg_create(n, *s["csr"])
        return s
    x = _xstar(n, gen)
    s["csr"], s["b"] = _matrix(case, gen, x)
    if case["do"] in ("solve", "spmv"):
        s["h"] = cg.cg_create(n, *s["csr"])
    if case["do"] == "spmv":
        s["x"] = x
    if case["do"] == "solve":
        if case["precond"] == "fsai":
            _check(cg.cg_fsai_load(s["h"], _weights()), s["h"])
        _check(cg.cg_prepare(s["h"], PRECOND[case["precond"]], PRECISION[case["precision"]]), s["h"])
    return s


def _batch(s, maxit):
    x = torch.zeros(s["total"], dtype=torch.float64, device="cuda")
    status, _, _ = cg.cg_solve_batch(s["h"], [s["b"][a:a + n] for a, n in s["starts"]], [x[a:a + n] for a, n in s["starts"]],
                                     TOL, maxit, cg.CG_PRECOND_JACOBI, PRECISION[s["case"]["precision"]])
    return x, status


def run(s):
    case = s["case"]
    if case["do"] == "batch":
        x, status = _batch(s, MAXIT)
        return {"x": x, "status": status}
    if case["do"] == "spmv":
        y = torch.empty_like(s["x"])
        _check(cg.cg_spmv(s["h"], s["x"], y), s["h"])
        return {"y": y}
    if case["do"] == "train":
        grad = torch.empty_like(s["params"])
        status, loss = cg.cg_fsai_loss_grad(s["h"], s["params"], grad, s["resid"], 0.1)
        _check(status, s["h"])
        return {"grad": grad, "loss": loss}
    x = torch.zeros_like(s["b"])
    if case["do"] == "noalloc":
        status, _, _ = cg.cg_solve_noalloc(*s["csr"], s["b"], x, TOL, MAXIT, PRECOND[case["precond"]])
        return {"x": x, "status": status}
    h = s["h"] if case["do"] == "solve" else cg.cg_create(s["b"].numel(), *s["csr"])
    if case["do"] == "fresh" and case["precond"] == "fsai":
        _check(cg.cg_fsai_classic(h), h)
    status, _, _ = cg.cg_solve(h, s["b"], x, TOL, MAXIT, PRECOND[case["precond"]], PRECISION[case["precision"]])
    if case["do"] == "fresh":
        cg.cg_destroy(h)
    return {"x": x, "status": status}


# ---------------------------------------------------------------- what a pass needs

L2_BYTES = 126e6


def _entries(case, side):
    if case["matrix"] == "graph":
        return 6.0 * case["n"]
    if case["matrix"] == "grid2d":
        return float(case["points"]) * side ** 2
    return 9.0 * side ** 2 if case["matrix"] == "q1" else float(case["points"]) * side ** 3


def _solve_work(n, nnz, precond, precision, shift):
    """A conjugate-gradient solve: an estimate of its steps from the condition number (about 2 / shift), each step's
    multiply-adds, and the bytes: the matrix and vectors once, or once a step where they exceed the L2."""
    cond = 2.0 / max(shift, 5e-4)
    steps = 0.5 * math.sqrt(cond) * math.log(2.0 / TOL) * 0.6 * (0.5 if precond == "fsai" else 1.0)
    v = 8.0 if precision == "fp64" else 4.0
    factor = 1.1 * nnz if precond == "fsai" else 0.0
    a_step = v * (nnz + factor) + 10.0 * v * n
    once = 12.0 * nnz + 20.0 * n
    return {"bytes": max(once, steps * a_step if v * (nnz + 4 * n) > L2_BYTES else once),
            "flops": steps * (2.0 * (nnz + factor) + 10.0 * n)}


def work(case):
    if case["do"] == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for side, points, _ in _members(case, 0):
            w = _solve_work(side ** 2, points * side ** 2, "jacobi", case["precision"], case["shift"])
            total = {k: total[k] + w[k] for k in total}
        return total
    n = _rows(case)
    nnz = _entries(case, case.get("side", 0))
    if case["do"] == "spmv":
        return {"bytes": 12.0 * nnz + 20.0 * n, "flops": 2.0 * nnz}
    if case["do"] == "train":
        tril = 5.0 * n  # 32-64-64-1 network, forward and twice that backward, three residuals
        return {"bytes": 12.0 * nnz + 28.0 * n + 8.0 * cg.CG_MLP_PARAMS, "flops": 6.0 * tril * cg.CG_MLP_PARAMS}
    return _solve_work(n, nnz, case["precond"], case["precision"], case.get("shift", 3e-3))


# ---------------------------------------------------------------- the results in 64 bits

def _bf16(t):
    return t.to(torch.bfloat16).to(torch.float64)


def _exact_train(case, seed):
    """The training loss and its gradient: the network's bf16 inputs and rounding points as stated in the library's
    header, everything else in 64 bits."""
    s = prepare(case, seed)
    deltas, vals, mask = s["table"]
    n, d = vals.shape[0], vals[:, 4]
    i = torch.arange(n, device="cuda")
    at = [(i + k).clamp(0, n - 1) for k in deltas]
    scaled = torch.stack([torch.where(mask[:, k], vals[:, k] / torch.sqrt(d * d[at[k]]), 0.0) for k in range(9)], 1)
    rows, slots = torch.nonzero(mask[:, :5], as_tuple=True)  # tril entries in CSR order
    cols = rows + torch.tensor(deltas, device="cuda")[slots]
    F = torch.zeros((rows.numel(), 32), dtype=torch.float64, device="cuda")
    F[torch.arange(rows.numel(), device="cuda"), slots] = 1.0
    F[:, 8], F[:, 9] = scaled[rows, slots], torch.log(d[cols] / d[rows])
    F[:, 10:19], F[:, 19:28], F[:, 28] = scaled[rows], scaled[cols], 1.0
    p = _bf16(s["params"])
    W1, b1, W2, b2, W3, b3 = (t.reshape(-1, k) if k > 1 else t for t, k in zip(
        torch.split(p, [2048, 64, 4096, 64, 64, 1]), (32, 1, 64, 1, 1, 1)))
    X = _bf16(F)
    z1 = X @ W1.T + b1
    h1 = _bf16(z1.clamp_min(0.0))
    z2 = h1 @ W2.T + b2
    h2 = z2.clamp_min(0.0)
    out = (h2 @ W3 + b3).requires_grad_(True)
    # the loss of G, differentiated down to the network's output
    on = rows == cols
    c0 = math.log(math.e - 1.0)
    g = torch.where(on, torch.nn.functional.softplus(out + c0, threshold=1000.0), out) / torch.sqrt(d[cols])
    G = torch.zeros((n, 5), dtype=torch.float64, device="cuda").index_put((rows, slots), g)

    def times(table, x, ks):
        return sum(torch.where(mask[:, k], table[:, k] * x[at[k]], 0.0) for k in ks)

    # g_i^T A g_i: A between two columns of row i's pattern
    quad = torch.zeros((), dtype=torch.float64, device="cuda")
    place = {v: k for k, v in enumerate((dy, dx) for dy in (-1, 0, 1) for dx in (-1, 0, 1))}
    spot = list(place)
    for a in range(5):
        for b in range(5):
            o = (spot[b][0] - spot[a][0], spot[b][1] - spot[a][1])
            if o in place:
                k = place[o]
                quad = quad + (torch.where(mask[:, a] & mask[:, b] & mask[at[a], k], vals[at[a], k], 0.0) * G[:, a] * G[:, b]).sum()
    loss = torch.log(quad / n) - 2.0 / n * torch.log(G[:, 4]).sum()
    for r in s["resid"]:
        u = times(G, r, range(5))
        v = torch.zeros_like(u)
        for k in range(5):
            v = v.index_add(0, at[k], torch.where(mask[:, k], G[:, k] * u, 0.0))
        e = times(vals, v, range(9)) - r
        loss = loss + 0.1 / 3 * (e @ e) / (r @ r)
    loss.backward()
    do = out.grad
    dz2 = do[:, None] * W3 * (z2 > 0)
    dz1 = (_bf16(dz2) @ W2) * (z1 > 0)
    grad = torch.cat([(_bf16(dz1).T @ X).reshape(-1), dz1.sum(0), (_bf16(dz2).T @ h1).reshape(-1), dz2.sum(0), h2.T @ do,
                      do.sum().reshape(1)])
    return {"grad": grad.detach(), "loss": float(loss.detach())}


def exact(case, seed):
    gen = _generator(seed)
    if case["do"] == "train":
        return _exact_train(case, seed)
    if case["do"] == "batch":
        parts = []
        for side, _, _ in _members(case, seed):
            parts.append(_xstar(side * side, gen))
            parts.append(torch.zeros(side * side % 2, dtype=torch.float64, device="cuda"))
        return {"x": torch.cat(parts), "status": None}
    x = _xstar(_rows(case), gen)
    if case["do"] == "spmv":
        return {"y": _matrix(case, gen, x)[1]}
    return {"x": x, "status": None}
