"""Workloads of the triangular solver as a user's program runs them, through its
public entry points: what each stands for, its inputs, one pass, the work it
cannot do without and the result in 64 bits by plain torch.

A case's ``kind`` names the program:

* ``solve``     one solve or adjoint solve on a kept plan (one or several
                right-hand sides);
* ``pair``      L then U, the preconditioner step ``z = U^{-1} L^{-1} r``;
* ``tuned``     the documented flow for a new matrix: tune once, then solve
                with ``algo="auto"``;
* ``values``    new values on a kept pattern, then a solve (a Newton or time
                step that refactors);
* ``autograd``  a differentiable solve, forward and backward;
* ``refined``   FP32 solves with FP64 refinement;
* ``batch``     many independent systems in one graph replay;
* ``setup``     a matrix that is used once: analysis, layout and one solve.

Matrices: ``ilu`` (ILU(0) factors of the 3-D 7-point operator with a seeded
reaction term), ``grid`` (triangles of the 5/9-point 2-D and 7/27-point 3-D
operators) and ``general`` (power-law row lengths, 70 % of the columns in a
band of 512).  Launch shapes are those a tuner run leaves behind for the
family (``autotune.apply_choice``); no shape means the plan's defaults.
"""
from __future__ import annotations

import math

import torch

from paper_1710_04985_gb300 import TriangularPlan, autotune, sparse_triangular_solve
from paper_1710_04985_gb300.batch import BatchedTriangularSolve

DEV = "cuda"
MAXLEN = 2000


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: a 2-D grid of a few thousand points, plan defaults;
        # launches and the latency of 127 dependent levels are all there is
        {"name": "grid5_64x64", "kind": "solve", "matrix": "grid", "dims": "64x64", "points": 5,
         "upper": False, "dtype": "f64", "algo": "self", "nrhs": 1, "transpose": False},
        # an ordinary adjoint solve on a ragged 3-D grid, plan defaults
        {"name": "grid7_61x47x53_adjoint", "kind": "solve", "matrix": "grid", "dims": "61x47x53",
         "points": 7, "upper": False, "dtype": "f64", "algo": "self", "nrhs": 1,
         "transpose": True},
        # the headline workload: applying an ILU(0) preconditioner of the 128^3 grid
        {"name": "ilu_128_pair", "kind": "pair", "matrix": "ilu", "dims": "128x128x128",
         "points": 7, "dtype": "f64", "algo": "partitioned", "lanes": 1, "block": 512,
         "part_rows": 16384, "cluster": 4},
        # the 2-D model problem in single precision, odd sides, 9-point rows:
        # thousands of levels of a few hundred rows
        {"name": "grid9_1021x1023_pair_f32", "kind": "pair", "matrix": "grid",
         "dims": "1021x1023", "points": 9, "dtype": "f32", "algo": "partitioned", "lanes": 4,
         "block": 512, "part_rows": 8192, "cluster": 4},
        # a general matrix of ordinary size, tuned once as the documents say
        {"name": "general_150k_tuned", "kind": "tuned", "matrix": "general", "n": 150001,
         "upper": False, "dtype": "f64"},
        # a solver layer in a training loop: the largest work of one pass, plan defaults
        {"name": "general_1m_autograd", "kind": "autograd", "matrix": "general", "n": 1000000,
         "upper": False, "dtype": "f64", "algo": "self"},
        # many right-hand sides at once (block Krylov methods)
        {"name": "ilu_128_k32", "kind": "solve", "matrix": "ilu", "dims": "128x128x128",
         "points": 7, "upper": False, "dtype": "f64", "algo": "self", "nrhs": 32,
         "transpose": False},
        # a few right-hand sides, single precision, upper factor, ragged grid, on the
        # level-ordered copy
        {"name": "ilu_97x101x89_k5_f32_upper", "kind": "solve", "matrix": "ilu",
         "dims": "97x101x89", "points": 7, "upper": True, "dtype": "f32", "algo": "permuted",
         "nrhs": 5, "transpose": False},
        # many independent systems of uneven size in one launch
        {"name": "batch_128_systems", "kind": "batch", "count": 128, "nmin": 1000, "nmax": 65536,
         "upper": False, "dtype": "f64", "algo": "partitioned", "lanes": 16, "block": 1024,
         "part_rows": 16384, "cluster": 1},
        # mixed precision: FP32 solves refined to FP64 accuracy
        {"name": "ilu_128_refined", "kind": "refined", "matrix": "ilu", "dims": "128x128x128",
         "points": 7, "upper": False, "dtype": "f64", "algo": "partitioned", "lanes": 1,
         "block": 512, "part_rows": 16384, "cluster": 4},
        # a matrix that is solved with once: the setup counts
        {"name": "ilu_128_setup", "kind": "setup", "matrix": "ilu", "dims": "128x128x128",
         "points": 7, "upper": False, "dtype": "f64", "algo": "self"},
        # new values every step on a kept pattern, long rows, upper triangle
        {"name": "grid27_61x47x53_values", "kind": "values", "matrix": "grid",
         "dims": "61x47x53", "points": 27, "upper": True, "dtype": "f64", "algo": "permuted"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dims(rng, points, nmin, nmax):
    """Sides of a grid of nmin..nmax points (log-uniform), up to 8 : 1."""
    d = 2 if points in (5, 9) else 3
    side = _log(rng, nmin, nmax) ** (1.0 / d)
    asp = [math.exp(rng.uniform(-math.log(2), math.log(2))) for _ in range(d)]
    g = math.prod(asp) ** (1.0 / d)
    return "x".join(str(max(8, int(side * a / g))) for a in asp)


def draw(rng):
    kind = rng.choice(["solve", "solve", "pair", "pair", "tuned", "autograd", "many", "batch",
                       "refined", "setup", "values"])
    dtype = rng.choice(["f64", "f64", "f32"])
    upper = rng.random() < 0.5
    grid = {"matrix": "grid", "points": rng.choice([5, 9, 7, 27])}
    if rng.random() < 0.4:
        grid = {"matrix": "ilu", "points": 7}

    def sized(nmin, nmax):
        return {**grid, "dims": _dims(rng, grid["points"], nmin, nmax)}

    def shape():
        # what the tuner leaves for a stencil: one lane a row for 5 and 7 points
        return {"algo": "partitioned", "lanes": {5: 1, 7: 1, 9: 4, 27: 8}[grid["points"]],
                "block": 512, "part_rows": rng.choice([0, 8192, 16384]),
                "cluster": rng.choice([1, 4])}

    if kind == "solve":
        c = sized(3000, 1500000)
        if rng.random() < 0.3:
            c = {"matrix": "general", "n": _log(rng, 3000, 400000)}
        return {"kind": "solve", **c, "upper": upper, "dtype": dtype,
                "algo": rng.choice(["self", "self", "permuted"]), "nrhs": 1,
                "transpose": rng.random() < 0.3}
    if kind == "pair":
        return {"kind": "pair", **sized(100000, 2000000), "dtype": dtype, **shape()}
    if kind == "tuned":
        return {"kind": "tuned", "matrix": "general", "n": _log(rng, 20000, 150000),
                "upper": upper, "dtype": dtype}
    if kind == "autograd":
        return {"kind": "autograd", "matrix": "general", "n": _log(rng, 30000, 900000),
                "upper": upper, "dtype": dtype, "algo": "self"}
    if kind == "many":
        return {"kind": "solve", **sized(30000, 1500000), "upper": upper, "dtype": dtype,
                "algo": rng.choice(["self", "permuted"]), "nrhs": rng.randint(2, 32),
                "transpose": rng.random() < 0.3}
    if kind == "batch":
        return {"kind": "batch", "count": _log(rng, 16, 128), "nmin": 1000,
                "nmax": _log(rng, 8000, 65536), "upper": upper, "dtype": dtype,
                "algo": "partitioned", "lanes": rng.choice([4, 8, 16]), "block": 1024,
                "part_rows": rng.choice([0, 16384]), "cluster": 1}
    if kind == "refined":
        return {"kind": "refined", **sized(100000, 2000000), "upper": upper, "dtype": "f64",
                **shape()}
    if kind == "setup":
        c = sized(30000, 2000000)
        if rng.random() < 0.3:
            c = {"matrix": "general", "n": _log(rng, 30000, 400000)}
        return {"kind": "setup", **c, "upper": upper, "dtype": dtype, "algo": "self"}
    return {"kind": "values", **sized(30000, 1500000), "upper": upper, "dtype": dtype,
            "algo": rng.choice(["permuted", "partitioned"])}


# ------------------------------------------------------------------ matrices
_OFFSETS = {
    5: [(0, -1), (-1, 0), (0, 0), (1, 0), (0, 1)],
    7: [(0, 0, -1), (0, -1, 0), (-1, 0, 0), (0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1)],
    9: [(x, y) for y in (-1, 0, 1) for x in (-1, 0, 1)],
    27: [(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)],
}


def _sides(case):
    return tuple(int(v) for v in case["dims"].split("x"))


def _grid_pattern(dims, points, upper):
    """(rowptr, colidx, rows) of one triangle, diagonal stored, x fastest."""
    n = math.prod(dims)
    lin = torch.arange(n, device=DEV)
    coords, rest = [], lin
    for d in dims:
        coords.append(rest % d)
        rest = rest // d
    strides = [math.prod(dims[:a]) for a in range(len(dims))]
    offs = sorted((sum(o * s for o, s in zip(off, strides)), off) for off in _OFFSETS[points])
    offs = [t for t in offs if (t[0] >= 0 if upper else t[0] <= 0)]
    cols = torch.empty(n, len(offs), dtype=torch.int32, device=DEV)
    keep = torch.ones(n, len(offs), dtype=torch.bool, device=DEV)
    for s, (delta, off) in enumerate(offs):
        cols[:, s] = lin + delta
        for a, o in enumerate(off):
            if o:
                c = coords[a] + o
                keep[:, s] &= (c >= 0) & (c < dims[a])
    rowptr = torch.zeros(n + 1, dtype=torch.int32, device=DEV)
    rowptr[1:] = keep.sum(1).cumsum(0)
    rows = lin[:, None].expand(-1, len(offs))[keep]
    return rowptr, cols[keep], rows


def _ilu_pivots(dims, diag):
    """Pivots of ILU(0) of the 7-point operator with diagonal ``diag``, plane
    x + y + z = const by plane."""
    nx, ny, nz = dims
    n = nx * ny * nz
    lin = torch.arange(n, device=DEV)
    x, y, z = lin % nx, (lin // nx) % ny, lin // (nx * ny)
    plane = x + y + z
    order = torch.sort(plane, stable=True)[1]
    ends = torch.bincount(plane).cumsum(0).tolist()
    inv = torch.zeros(n + 1, dtype=torch.float64, device=DEV)   # 1/pivot; slot n: none
    none = torch.full_like(lin, n)
    nb = torch.stack([torch.where(x > 0, lin - 1, none), torch.where(y > 0, lin - nx, none),
                      torch.where(z > 0, lin - nx * ny, none)])[:, order]
    d = diag[order]
    first = 0
    for end in ends:
        inv[order[first:end]] = 1.0 / (d[first:end] - inv[nb[:, first:end]].sum(0))
        first = end
    return 1.0 / inv[:n]


def _general_entries(n):
    """Stored entries of a general matrix: 13 off-diagonals a row on average."""
    return 14 * n


def _general(n, gen):
    """Lower triangle with power-law row lengths, diagonally dominant, of
    _general_entries(n) entries: lengths are stratified draws of the Pareto law
    (shape 2, scale 8, at most MAXLEN), repeated columns are dropped, and what
    is then over the count is dropped at random."""
    i = torch.arange(n, device=DEV)
    u = (torch.randperm(n, generator=gen, device=DEV) +
         torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)) / n
    length = (8.0 / u.clamp(min=1e-9).sqrt()).round().to(torch.int64).clamp(max=MAXLEN)
    m = torch.minimum(length, i + 1) - 1
    r = torch.repeat_interleave(i, m)
    band = torch.rand(r.numel(), generator=gen, device=DEV) < 0.7
    t = torch.rand(r.numel(), generator=gen, device=DEV, dtype=torch.float64)
    lo = torch.where(band, (r - 512).clamp(min=0), torch.zeros_like(r))
    c = torch.minimum(lo + (t * (r - lo)).to(torch.int64), r - 1)
    keys = torch.unique(r * n + c)
    want = _general_entries(n) - n
    assert keys.numel() >= want, (n, keys.numel(), want)
    keys = keys[torch.randperm(keys.numel(), generator=gen, device=DEV)[:want]]
    keys = torch.cat([keys, i * n + i]).sort()[0]
    rows = keys // n
    cols = keys - rows * n
    off = rows != cols
    # values of 20 bits after the point: their sums are exact in any order, so a
    # seed always gives the same diagonal
    q = torch.randint(-(1 << 20), (1 << 20) + 1, (keys.numel(),), generator=gen, device=DEV)
    vals = torch.where(off, q, 0).to(torch.float64) / (1 << 20)
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = torch.bincount(rows, minlength=n).cumsum(0)
    csum = torch.cat([torch.zeros_like(rowptr[:1]), torch.where(off, q.abs(), 0).cumsum(0)])
    total = (csum[rowptr[1:]] - csum[rowptr[:-1]]).to(torch.float64) / (1 << 20)
    vals = torch.where(off, vals, (1.0 + total)[rows])
    return rowptr.to(torch.int32), cols.to(torch.int32), vals, rows


def _reversed(rowptr, colidx, vals, rows):
    """The upper triangle obtained by reversing the order of the unknowns."""
    n = rowptr.numel() - 1
    lens = (rowptr[1:] - rowptr[:-1]).flip(0)
    rp = torch.zeros_like(rowptr)
    rp[1:] = lens.cumsum(0)
    return rp, (n - 1 - colidx).flip(0).contiguous(), vals.flip(0).contiguous(), \
        (n - 1 - rows).flip(0).contiguous()


def _matrix(case, upper, gen):
    """(rowptr, colidx, vals, rows, unit) of the case's matrix in FP64."""
    if case["matrix"] == "general":
        m = _general(case["n"], gen)
        return (*(_reversed(*m) if upper else m), False)
    dims, points = _sides(case), case["points"]
    rowptr, colidx, rows = _grid_pattern(dims, points, upper)
    n = rowptr.numel() - 1
    # a reaction term of up to 5 % of the diagonal, seeded
    react = torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)
    diag = (points - 1) * (1.0 + 0.05 * react)
    on = rows == colidx
    if case["matrix"] == "ilu":
        piv = _ilu_pivots(dims, diag)
        if upper:
            return rowptr, colidx, torch.where(on, piv[rows], -1.0), rows, False
        return rowptr, colidx, torch.where(on, 1.0, -1.0 / piv[colidx.long()]), rows, True
    return rowptr, colidx, torch.where(on, diag[rows], -1.0), rows, False


def _batch_sizes(case):
    """Log-uniform sizes, one from each of ``count`` equal strata."""
    lo, hi, k = math.log(case["nmin"]), math.log(case["nmax"]), case["count"]
    return [int(round(math.exp(lo + (s + 0.5) / k * (hi - lo)))) for s in range(k)]


def _batch_systems(case, gen):
    sizes = _batch_sizes(case)
    out = []
    for s in torch.randperm(len(sizes), generator=gen, device=DEV).tolist():
        m = _general(sizes[s], gen)
        out.append((_reversed(*m) if case["upper"] else m)[:3])
    return out


def _dtype(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _rhs(n, nrhs, gen, dtype):
    shape = (n,) if nrhs == 1 else (n, nrhs)
    return (2 * torch.rand(shape, generator=gen, device=DEV, dtype=torch.float64) - 1).to(dtype)


def _inputs(case, seed):
    """Matrices (in the case's type) and vectors of a case, from the seed alone."""
    gen = _gen(seed)
    dtype = _dtype(case)
    if case["kind"] == "batch":
        systems = [(rp, ci, va.to(dtype)) for rp, ci, va in _batch_systems(case, gen)]
        n = sum(rp.numel() - 1 for rp, _, _ in systems)
        return {"systems": systems, "b": _rhs(n, 1, gen, dtype)}
    ups = (False, True) if case["kind"] == "pair" else (case["upper"],)
    s = {"mats": []}
    for upper in ups:
        rp, ci, va, rows, unit = _matrix(case, upper, gen)
        s["mats"].append({"rowptr": rp, "colidx": ci, "vals": va.to(dtype), "rows": rows,
                          "upper": upper, "unit": unit})
    n = s["mats"][0]["rowptr"].numel() - 1
    s["b"] = _rhs(n, case.get("nrhs", 1), gen, dtype)
    if case["kind"] == "autograd":
        s["g"] = _rhs(n, 1, gen, dtype)
    if case["kind"] == "values":
        # the next step's values: every stored value scaled by up to 5 %
        scale = 1.0 + 0.05 * torch.rand(ci.numel(), generator=gen, device=DEV,
                                        dtype=torch.float64)
        s["vals2"] = torch.where(rows == ci, va * 1.05, va * scale / 1.05).to(dtype)
    return s


# ------------------------------------------------------------------ one pass
def _plan(m):
    return TriangularPlan(m["rowptr"], m["colidx"], m["vals"], upper=m["upper"], unit=m["unit"])


def _shape(case, plan):
    if "lanes" in case:
        autotune.apply_choice(plan, [case["algo"], case["lanes"], case["block"], 0,
                                     case["part_rows"], case["cluster"]])


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    kind = case["kind"]
    if kind == "batch":
        s["batch"] = BatchedTriangularSolve(s.pop("systems"), upper=case["upper"],
                                            dtype=_dtype(case), device=DEV, tune=False)
        _shape(case, s["batch"].plan)
        s["batch"].capture()
        return s
    if kind == "setup":
        return s
    s["plans"] = [_plan(m) for m in s["mats"]]
    for p in s["plans"]:
        _shape(case, p)
        if kind == "tuned":
            autotune.tune_algos(p, s["b"], quick=True, use_cache=False)
        elif kind == "autograd":
            p.prepare_transpose()
        elif kind in ("solve", "values", "pair"):
            p.prepare(case["algo"], transpose=case.get("transpose", False))
    if kind == "autograd":
        s["vals"] = s["mats"][0]["vals"].requires_grad_(True)
        s["b"].requires_grad_(True)
    s["x"] = torch.empty_like(s["b"])
    if kind == "pair":
        s["y"] = torch.empty_like(s["b"])
    return s


def run(state):
    s, case = state, state["case"]
    kind = case["kind"]
    if kind == "batch":
        return s["batch"].solve(s["b"])
    if kind == "setup":
        m = s["mats"][0]
        with _plan(m) as p:
            x = p.solve(s["b"], algo=case["algo"])
            lev = p.levels()
            return {"x": x, "lev": lev["lev"], "jlev": lev["jlev"], "nlev": lev["nlev"]}
    p = s["plans"][0]
    if kind == "solve":
        if case["transpose"]:
            return p.solve_transpose(s["b"], out=s["x"], algo=case["algo"])
        return p.solve(s["b"], out=s["x"], algo=case["algo"])
    if kind == "pair":
        y = p.solve(s["b"], out=s["y"], algo="auto")
        return {"y": y, "x": s["plans"][1].solve(y, out=s["x"], algo="auto")}
    if kind == "tuned":
        return p.solve(s["b"], out=s["x"], algo="auto")
    if kind == "values":
        p.set_values(s["vals2"])
        return p.solve(s["b"], out=s["x"], algo=case["algo"])
    if kind == "refined":
        x, iters, _ = p.solve_refined(s["b"], out=s["x"])
        return {"x": x, "iters": iters}
    x = sparse_triangular_solve(p, s["vals"], s["b"], algo=case["algo"])
    gv, gb = torch.autograd.grad(x, (s["vals"], s["b"]), s["g"])
    return {"x": x.detach(), "grad_vals": gv, "grad_b": gb}


# ------------------------------------------------------------------ work, exact
def _entries(case):
    """(n, stored entries) of one matrix of the case."""
    if case["kind"] == "batch":
        sizes = _batch_sizes(case)
        return sum(sizes), sum(_general_entries(n) for n in sizes)
    if case["matrix"] == "general":
        return case["n"], _general_entries(case["n"])
    dims = _sides(case)
    n = math.prod(dims)
    nnz = 0
    for off in _OFFSETS[case["points"]]:
        nnz += math.prod(d - abs(o) for d, o in zip(dims, off))
    return n, (nnz + n) / 2


def work(case):
    n, nnz = _entries(case)
    e = 8 if case["dtype"] == "f64" else 4
    k = case.get("nrhs", 1)
    matrix = nnz * (4 + e) + 4 * n            # columns, values, row pointers
    solve = matrix + 2 * n * e * k
    flops = 2 * nnz * k
    kind = case["kind"]
    if kind == "pair":
        return {"bytes": 2 * solve, "flops": 2 * flops}
    if kind == "autograd":                    # forward, adjoint, gradient of every entry
        return {"bytes": 2 * solve + nnz * (4 + e) + 2 * n * e, "flops": 5 * nnz}
    if kind == "refined":                     # matrix in both precisions, b, x
        return {"bytes": matrix + 4 * nnz + 16 * n, "flops": 4 * nnz}
    if kind == "setup":                       # the solve and the level arrays
        return {"bytes": solve + 8 * n, "flops": flops}
    return {"bytes": solve, "flops": flops}


def _solve64(m, b, transpose=False):
    """The substitution's result in FP64: x = (b - (A - D) x) / D repeated until
    nothing changes (level l is final after l + 1 steps)."""
    n = m["rowptr"].numel() - 1
    rows, cols, vals = m["rows"], m["colidx"].long(), m["vals"].double()
    on = rows == cols
    if m["unit"]:
        d = torch.ones(n, dtype=torch.float64, device=DEV)
    else:
        d = torch.zeros(n, dtype=torch.float64, device=DEV)
        d[rows[on]] = vals[on]
    i, j = (cols, rows) if transpose else (rows, cols)
    off = torch.sparse_coo_tensor(torch.stack([i[~on], j[~on]]), vals[~on],
                                  (n, n)).coalesce().to_sparse_csr()
    rhs = (b.double() if b.dim() == 2 else b.double()[:, None])
    x = rhs / d[:, None]
    for step in range(n):
        new = (rhs - off @ x) / d[:, None]
        done = step % 16 == 15 and torch.equal(new, x)
        x = new
        if done or step >= 4000:
            break
    return x if b.dim() == 2 else x[:, 0]


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "batch":
        out, at = [], 0
        for rp, ci, va in s["systems"]:
            n = rp.numel() - 1
            rows = torch.repeat_interleave(torch.arange(n, device=DEV), (rp[1:] - rp[:-1]).long())
            out.append(_solve64({"rowptr": rp, "colidx": ci, "vals": va, "rows": rows,
                                 "unit": False}, s["b"][at:at + n]))
            at += n
        return torch.cat(out)
    m = s["mats"][0]
    if kind == "values":
        m = {**m, "vals": s["vals2"]}
    x = _solve64(m, s["b"], case.get("transpose", False))
    if kind == "pair":
        # U is solved for the rounded y, as any program does; its own rounding
        # is far below the bounds in either type
        return {"y": x, "x": _solve64(s["mats"][1], x)}
    if kind == "refined":
        return {"x": x, "iters": None}
    if kind == "setup":
        return {"x": x, "lev": None, "jlev": None, "nlev": None}
    if kind == "autograd":
        y = _solve64(m, s["g"], transpose=True)
        return {"x": x, "grad_vals": -y[m["rows"]] * x[m["colidx"].long()], "grad_b": y}
    return x
