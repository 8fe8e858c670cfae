"""The workloads that the library's speed is judged by, from the smallest product to whole solves.

Every case goes through the public Python entry points (``packsell_*`` and ``autograd``). The matrices
are the shapes that the benchmark and the tests use, built here on the GPU from a seed: 5-point and
27-point stencils, variable-coefficient Poisson problems, and power-law ("irregular") matrices.

A case names its ``kind`` (what the program does) and its matrix:

* ``spmv``, ``spmm``: y = A x and Y = A X with a matrix encoded once, the library's main use;
* ``batch``: the products of many small matrices by one plan;
* ``train``: the forward product and both gradients, one step of a training loop;
* ``encode``: new CSR values into a packed matrix, and the first product with it;
* ``pcg``: inner-outer CG on operators that are kept, one right-hand side after another;
* ``diff``: a differentiable solve, which encodes, solves and solves the adjoint system;
* ``f3r``: the nested FGMRES solver.
"""
from __future__ import annotations

import math

import torch

from paper_2604_13433_gb300 import autograd as ag
from paper_2604_13433_gb300 import packsell as ps

DEV = "cuda"
ZIPF_MAX = 4096  # longest row of the power-law matrices


# ---------------------------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------------------------
def _spmv(name, matrix, **kw):
    return dict({"name": name, "kind": "spmv", "matrix": matrix, "C": 32, "sigma": 256, "fmt": "fp16",
                 "D": 15, "explicit": False}, **kw)


def listed():
    return [
        # the smallest product: a 64 x 64 Laplacian, where the call and the launch are all there is
        _spmv("spmv_poisson5_64", "stencil5", nx=64, ny=64, nz=1),
        # the headline product: the HPCG 7_7_7 pattern, FP16 values, rows left in storage order
        _spmv("spmv_stencil27_128", "stencil27", nx=128, ny=128, nz=128, explicit=True),
        # a large power-law graph or circuit matrix in CSR order (an odd number of rows)
        _spmv("spmv_irregular_4M", "irregular", n=3999971, C=1, sigma=1),
        # a block of 16 vectors (block Krylov, multi-scenario) through the same stencil matrix
        _spmv("spmm16_stencil27_128", "stencil27", kind="spmm", k=16, nx=128, ny=128, nz=128),
        # 64 feature columns through a ragged grid, with the more exact E8M11 values
        _spmv("spmm64_stencil27_ragged", "stencil27", kind="spmm", k=64, nx=101, ny=83, nz=117,
              fmt="e8my", D=11),
        # 64 feature columns through a power-law graph (a graph network's aggregation)
        _spmv("spmm64_irregular_1M", "irregular", kind="spmm", k=64, n=1000003, C=1, sigma=1),
        # 256 power-law matrices of 1,000 to 100,000 rows in one call
        {"name": "batch256_irregular", "kind": "batch", "count": 256, "nmin": 1000, "nmax": 100000,
         "k": 1},
        # one training step over a stencil operator: product, gradient of x and of the values
        _spmv("train_stencil27_112", "stencil27", kind="train", nx=113, ny=112, nz=111),
        # new values of a mid-sized operator: encode and use it
        _spmv("encode_stencil27_96", "stencil27", kind="encode", nx=97, ny=96, nz=95, fmt="e8my",
              D=11),
        # a 3-D variable-coefficient problem solved again for each new right-hand side
        {"name": "pcg_poisson7_192", "kind": "pcg", "nx": 192, "ny": 192, "nz": 192, "fmt": "fp16",
         "D": 15, "m_in": 50, "rtol": 1e-10},
        # 64 systems of 32^2 to 256^2 cells in one block-diagonal solve, with its gradients
        {"name": "diff_poisson5_x64", "kind": "diff", "count": 64, "lmin": 32, "lmax": 256,
         "fmt": "e8my", "D": 11, "m_in": 20, "rtol": 1e-12},
        # the nested solver on the scaled 27-point matrix
        {"name": "f3r_stencil27_128", "kind": "f3r", "nx": 128, "ny": 128, "nz": 128, "fmt": "fp16",
         "D": 15, "rtol": 1e-10},
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def _values(rng):
    return rng.choice([{"fmt": "fp16", "D": 15}, {"fmt": "e8my", "D": 15}, {"fmt": "e8my", "D": 11},
                       {"fmt": "e8my", "D": 7}])


def _grid(rng, lo, hi):
    """Three sides whose product is spread over [lo^3, hi^3]."""
    side = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    a, b = math.exp(rng.uniform(-0.25, 0.25)), math.exp(rng.uniform(-0.25, 0.25))
    d = [min(max(int(round(side * f)), lo // 2), 160) for f in (a, b, 1 / (a * b))]
    while d[0] * d[1] * d[2] > hi ** 3:
        d[d.index(max(d))] -= 1
    return {"nx": d[0], "ny": d[1], "nz": d[2]}


def _stencil_or_irregular(rng, n_lo, n_hi):
    if rng.random() < 0.5:
        return dict(matrix="stencil27", C=32, sigma=256,
                    **_grid(rng, round(n_lo ** (1 / 3)), min(128, round(n_hi ** (1 / 3)))))
    return dict(matrix="irregular", C=1, sigma=1, n=_log(rng, n_lo, n_hi))


def draw(rng):
    kind = rng.choice(["spmv", "spmv", "spmm", "spmm", "batch", "train", "encode", "pcg", "diff", "f3r"])
    if kind in ("spmv", "spmm", "train", "encode"):
        c = {"kind": kind, "explicit": False, **_values(rng)}
        if kind == "spmv" and rng.random() < 0.34:
            c.update(matrix="stencil5", C=32, sigma=256, nx=_log(rng, 33, 2048), ny=_log(rng, 33, 2048), nz=1)
        elif kind == "spmv":
            c.update(_stencil_or_irregular(rng, 30000, 4000000))
        elif kind == "spmm":
            c.update(_stencil_or_irregular(rng, 30000, 1000000), k=rng.choice([2, 4, 6, 8, 16, 24, 32, 48, 64]))
        else:
            c.update(_stencil_or_irregular(rng, 30000, 1400000))
        return c
    if kind == "batch":
        return {"kind": kind, "count": _log(rng, 16, 256), "nmin": _log(rng, 500, 2000),
                "nmax": _log(rng, 5000, 100000), "k": rng.choice([1, 1, 4, 16])}
    if kind == "pcg":
        return {"kind": kind, **_grid(rng, 40, 160), **_values(rng), "m_in": rng.choice([20, 50, 80]),
                "rtol": 1e-10}
    if kind == "diff":
        lmin = rng.randint(16, 48)
        return {"kind": kind, "count": _log(rng, 8, 64), "lmin": lmin, "lmax": rng.randint(lmin + 8, 256),
                "fmt": "e8my", "D": rng.choice([7, 11]), "m_in": rng.choice([10, 20, 40]), "rtol": 1e-12}
    return {"kind": kind, **_grid(rng, 40, 128), "fmt": "fp16", "D": 15, "rtol": 1e-10}


# ---------------------------------------------------------------------------------------------
# matrices (CSR on the GPU)
# ---------------------------------------------------------------------------------------------
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + salt)
    return g


def _uniform(g, n, lo=-1.0, hi=1.0, dtype=torch.float32):
    return torch.rand(n, generator=g, device=DEV, dtype=dtype) * (hi - lo) + lo


def _csr(cols, vals=None):
    """CSR of an [n, w] table of columns (-1: absent, else increasing in a row)."""
    ok = cols >= 0
    rowptr = torch.zeros(cols.shape[0] + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(ok.sum(1), 0, out=rowptr[1:])
    return rowptr, cols[ok].to(torch.int32), None if vals is None else vals[ok]


def _stencil_cols(nx, ny, nz, reach):
    """Columns of the (2 reach + 1)^d box (reach = (x, y, z)) or, for "cross", of the axis stencil."""
    n = nx * ny * nz
    i = torch.arange(n, device=DEV, dtype=torch.int32)
    x, y, z = i % nx, (i // nx) % ny, i // (nx * ny)
    offs = [(dx, dy, dz) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)
            if (reach == "box" or abs(dx) + abs(dy) + abs(dz) <= 1) and (nz > 1 or dz == 0)]
    cols = torch.empty((n, len(offs)), dtype=torch.int32, device=DEV)
    for k, (dx, dy, dz) in enumerate(offs):
        ok = (x + dx >= 0) & (x + dx < nx) & (y + dy >= 0) & (y + dy < ny) & (z + dz >= 0) & (z + dz < nz)
        cols[:, k] = torch.where(ok, i + (dz * nx * ny + dy * nx + dx), -1)
    return cols, offs


def _stencil(case, seed):
    """5-point (values 4, -1 times 1 + U(-0.1, 0.1)) or 27-point (26, -(1 + U(-0.1, 0.1))) matrix."""
    box = case["matrix"] == "stencil27"
    cols, offs = _stencil_cols(case["nx"], case["ny"], case["nz"], "box" if box else "cross")
    n, w = cols.shape
    rowptr, col, _ = _csr(cols)
    row = torch.repeat_interleave(torch.arange(n, device=DEV, dtype=torch.int32), rowptr.diff())
    val = -(1.0 + _uniform(_gen(seed, 1), col.numel(), -0.1, 0.1))
    val = torch.where(col == row, torch.full_like(val, 26.0 if box else 4.0), val)
    return n, n, rowptr, col, val


def _irregular(sizes, seed, pattern=None):
    """Block-diagonal concatenation of power-law matrices (Zipf(2) row lengths up to 4,096; columns 95 %
    normal around the diagonal, 5 % uniform; values N(0, 1)). Columns are local to each block; ``pattern``
    is the pattern's own seed where only the values are to change with ``seed``."""
    g = _gen(seed if pattern is None else pattern, 2)
    size = torch.tensor(sizes, device=DEV, dtype=torch.int64)
    n = int(sum(sizes))
    block = torch.repeat_interleave(torch.arange(len(sizes), device=DEV), size)
    first = torch.cumsum(size, 0) - size
    m = size[block]
    pos = torch.arange(n, device=DEV) - first[block]
    p = 1.0 / torch.arange(1, ZIPF_MAX + 1, device=DEV, dtype=torch.float64) ** 2
    cdf = torch.cumsum(p, 0) / p.sum()
    length = torch.searchsorted(cdf, torch.rand(n, generator=g, device=DEV, dtype=torch.float64)) + 1
    length = torch.minimum(length, torch.minimum(m, torch.full_like(m, ZIPF_MAX)))
    row = torch.repeat_interleave(torch.arange(n, device=DEV), length)

    def columns(r):
        spread = torch.clamp(m[r].double() / 8, max=1000.0)
        c = (pos[r] + torch.round(spread * torch.randn(r.numel(), generator=g, device=DEV)).long())
        u = (torch.rand(r.numel(), generator=g, device=DEV, dtype=torch.float64) * m[r]).long()
        c = torch.where(torch.rand(r.numel(), generator=g, device=DEV) < 0.05, u, c)
        return torch.minimum(torch.clamp(c, min=0), m[r] - 1)

    key = row * (1 << 23) + columns(row)
    for _ in range(8):  # repeated columns are drawn again, then what still repeats is left out
        key = key.sort().values
        dup = torch.zeros_like(key, dtype=torch.bool)
        dup[1:] = key[1:] == key[:-1]
        r = (key[dup] >> 23)
        if r.numel() == 0:
            break
        key[dup] = r * (1 << 23) + columns(r)
    key = torch.unique(key)
    row, col = key >> 23, (key & ((1 << 23) - 1)).to(torch.int32)
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(row, minlength=n), 0, out=rowptr[1:])
    val = torch.randn(col.numel(), generator=_gen(seed, 9), device=DEV)
    return rowptr, col, val


def _matrix(case, seed):
    if case["matrix"] == "irregular":  # a gradient has the pattern's size: a training loop keeps the pattern
        rowptr, col, val = _irregular([case["n"]], seed, 0 if case["kind"] == "train" else None)
        return case["n"], case["n"], rowptr, col, val
    return _stencil(case, seed)


def _scaled(n, rowptr, col, val):
    row = torch.repeat_interleave(torch.arange(n, device=DEV), rowptr.diff())
    at = col == row
    d = torch.ones(n, dtype=torch.float64, device=DEV)
    d[row[at]] = val[at].double()
    s = d.rsqrt()
    return val.double() * s[row] * s[col.long()]


def _poisson7(case, seed):
    """7-point variable-coefficient Poisson (face coefficients exp(N(0, 1)), Dirichlet), scaled to a
    unit diagonal, in FP64."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    g = _gen(seed, 3)

    def face(sz, sy, sx):
        return torch.exp(torch.randn((sz, sy, sx), generator=g, device=DEV, dtype=torch.float64))

    fx, fy, fz = face(nz, ny, nx + 1), face(nz, ny + 1, nx), face(nz + 1, ny, nx)
    diag = (fx[:, :, 1:] + fx[:, :, :-1] + fy[:, 1:] + fy[:, :-1] + fz[1:] + fz[:-1]).reshape(-1)
    coef = {(-1, 0, 0): fx[:, :, :-1], (1, 0, 0): fx[:, :, 1:], (0, -1, 0): fy[:, :-1],
            (0, 1, 0): fy[:, 1:], (0, 0, -1): fz[:-1], (0, 0, 1): fz[1:]}
    cols, offs = _stencil_cols(nx, ny, nz, "cross")
    s = diag.rsqrt()
    vals = torch.empty(cols.shape, dtype=torch.float64, device=DEV)
    for k, o in enumerate(offs):
        if o == (0, 0, 0):
            vals[:, k] = 1.0
        else:
            vals[:, k] = -coef[o].reshape(-1) * s * s[cols[:, k].clamp(min=0).long()]
    rowptr, col, val = _csr(cols, vals)
    return cols.shape[0], rowptr, col, val


def _systems(case, seed):
    """Block-diagonal 5-point variable-coefficient systems (coefficients exp(N(0, 0.5))) in FP64. The
    sides are the same for every seed; the coefficients are not."""
    span = case["lmax"] - case["lmin"] + 1
    sides = [case["lmin"] + (i * 7919 + 13) % span for i in range(case["count"])]
    g = _gen(seed, 4)
    L = torch.tensor(sides, device=DEV)
    size = L * L
    n = int(size.sum())
    b = torch.repeat_interleave(torch.arange(len(sides), device=DEV), size)
    loc = torch.arange(n, device=DEV) - (torch.cumsum(size, 0) - size)[b]
    Lc = L[b]
    r, c = loc // Lc, loc % Lc
    i = torch.arange(n, device=DEV)
    right, down, left, top = (torch.exp(0.5 * torch.randn(n, generator=g, device=DEV, dtype=torch.float64))
                              for _ in range(4))
    prev, above = (i - 1).clamp(min=0), (i - Lc).clamp(min=0)
    w = torch.where(c > 0, right[prev], left)
    u = torch.where(r > 0, down[above], top)
    cols = torch.stack([torch.where(r > 0, i - Lc, -1), torch.where(c > 0, i - 1, -1), i,
                        torch.where(c < Lc - 1, i + 1, -1), torch.where(r < Lc - 1, i + Lc, -1)], 1)
    vals = torch.stack([-u, -w, u + w + right + down, -right, -down], 1)
    rowptr, col, val = _csr(cols, vals)
    return n, rowptr, col, val


def _batch_sizes(case):
    lo, hi, cnt = math.log(case["nmin"]), math.log(case["nmax"]), case["count"]
    return [int(math.exp(lo + (hi - lo) * ((i * 7919 + 17) % cnt + 0.5) / cnt)) for i in range(cnt)]


def _rhs(n, seed):
    return _uniform(_gen(seed, 5), n, 0.0, 1.0, torch.float64)


def _input(case, m, seed):
    k = case.get("k", 1)
    return _uniform(_gen(seed, 6), m * k).view(m, k) if case["kind"] == "spmm" else _uniform(_gen(seed, 6), m)


def _encode(case, n, m, rowptr, col, val, **kw):
    return ps.packsell_encode(rowptr, col, val, n, m, C=case["C"], sigma=case["sigma"], D=case["D"],
                              fmt=case["fmt"], explicit_perm=case.get("explicit", False), **kw)


# ---------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("spmv", "spmm"):
        n, m, rowptr, col, val = _matrix(case, seed)
        return {"kind": kind, "A": _encode(case, n, m, rowptr, col, val), "x": _input(case, m, seed)}
    if kind == "train":
        n, m, rowptr, col, val = _matrix(case, seed)
        return {"kind": kind, "A": _encode(case, n, m, rowptr, col, val, keep_rowptr=True),
                "x": _input(case, m, seed).requires_grad_(True), "val": val.requires_grad_(True),
                "dy": _uniform(_gen(seed, 7), n)}
    if kind == "encode":
        n, m, rowptr, col, val = _matrix(case, seed)
        return {"kind": kind, "case": case, "csr": (n, m, rowptr, col, val), "x": _input(case, m, seed)}
    if kind == "batch":
        sizes, k = _batch_sizes(case), case["k"]
        rowptr, col, val = _irregular(sizes, seed)
        n = sum(sizes)
        X = _uniform(_gen(seed, 6), n * k).view(n, k)
        Y = torch.empty((n, k), device=DEV)
        ends = rowptr[torch.tensor([0] + sizes, device=DEV).cumsum(0)].tolist()
        mats, xs, ys, r0 = [], [], [], 0
        for i, s in enumerate(sizes):
            a, b = ends[i], ends[i + 1]
            mats.append(ps.packsell_encode(rowptr[r0:r0 + s + 1] - a, col[a:b], val[a:b], s, s, C=1, sigma=1,
                                           D=15, fmt="fp16"))
            xs.append(X[r0:r0 + s] if k > 1 else X[r0:r0 + s, 0])
            ys.append(Y[r0:r0 + s] if k > 1 else Y[r0:r0 + s, 0])
            r0 += s
        create = ps.packsell_batch_create if k == 1 else ps.packsell_batch_create_spmm
        return {"kind": kind, "plan": create(mats, xs, ys), "Y": Y}
    if kind == "pcg":
        n, rowptr, col, val = _poisson7(case, seed)
        return {"kind": kind, "b": _rhs(n, seed), "m_in": case["m_in"], "rtol": case["rtol"],
                "A": ps.packsell_encode(rowptr, col, val, n, n, fmt="sell_f64"),
                "Ain": ps.packsell_encode(rowptr, col, val, n, n, fmt=case["fmt"], D=case["D"])}
    if kind == "diff":
        n, rowptr, col, val = _systems(case, seed)
        return {"kind": kind, "rowptr": rowptr, "col": col, "val": val.requires_grad_(True),
                "b": _rhs(n, seed).requires_grad_(True),
                "g": _uniform(_gen(seed, 8), n, 0.0, 1.0, torch.float64),
                "opts": {k: case[k] for k in ("fmt", "D", "m_in", "rtol")}}
    n, m, rowptr, col, val = _stencil(dict(case, matrix="stencil27"), seed)
    val = _scaled(n, rowptr, col, val)
    A = [ps.packsell_encode(rowptr, col, val, n, n, fmt=f, D=case["D"])
         for f in ("sell_f64", "sell_f32", case["fmt"])]
    return {"kind": kind, "A": A, "b": _rhs(n, seed), "rtol": case["rtol"]}


def run(s):
    kind = s["kind"]
    if kind == "spmv":
        return ps.packsell_spmv(s["A"], s["x"])
    if kind == "spmm":
        return ps.packsell_spmm(s["A"], s["x"])
    if kind == "batch":
        (ps.packsell_batch_spmv if isinstance(s["plan"], ps.PackSELLBatch) else ps.packsell_batch_spmm)(s["plan"])
        return s["Y"]
    if kind == "train":
        y = ag.spmv(s["A"], s["x"], s["val"])
        dval, dx = torch.autograd.grad(y, (s["val"], s["x"]), s["dy"])
        return {"y": y.detach(), "dx": dx, "dval": dval}
    if kind == "encode":
        A = _encode(s["case"], *s["csr"], keep_rowptr=True)
        return {"y": ps.packsell_spmv(A, s["x"]), "words": A.n_words, "dummies": A.n_dummies, "pad": A.n_pad}
    if kind == "pcg":
        return ps.packsell_pcg(s["A"], s["b"], A_inner=s["Ain"], m_in=s["m_in"], rtol=s["rtol"])[0]
    if kind == "diff":
        x = ag.solve(s["rowptr"], s["col"], s["val"], s["b"], **s["opts"])
        dval, db = torch.autograd.grad(x, (s["val"], s["b"]), s["g"])
        return {"x": x.detach(), "dval": dval, "db": db}
    return ps.packsell_f3r(*s["A"], s["b"], rtol=s["rtol"])[0]


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------
def _mean_length(limit):
    top = min(ZIPF_MAX, limit)
    p = [1.0 / k ** 2 for k in range(1, ZIPF_MAX + 1)]
    return sum(min(k, top) * q for k, q in enumerate(p, 1)) / sum(p)


def _size(case):
    """(rows, nonzeros); expected nonzeros for a power-law matrix."""
    if case.get("matrix") == "irregular":
        return case["n"], case["n"] * _mean_length(case["n"])
    if case["kind"] == "batch":
        s = _batch_sizes(case)
        return sum(s), sum(v * _mean_length(v) for v in s)
    if case["kind"] == "diff":
        span = case["lmax"] - case["lmin"] + 1
        L = [case["lmin"] + (i * 7919 + 13) % span for i in range(case["count"])]
        return sum(v * v for v in L), sum(5 * v * v - 4 * v for v in L)
    x, y, z = case["nx"], case["ny"], case["nz"]
    n = x * y * z
    if case["kind"] == "pcg":
        return n, 7 * n - 2 * (x * y + y * z + x * z)
    if case.get("matrix") == "stencil5":
        return n, 5 * n - 2 * (x + y)
    return n, (3 * x - 2) * (3 * y - 2) * (3 * z - 2)


def work(case):
    """Stored nonzeros as 4-byte words, each input vector read once, each output written once; CSR
    inputs as they are given. A solve counts one reading of its operators and vectors and one product
    with each: how often an iteration needs them is the method's choice."""
    n, nnz = _size(case)
    kind, k = case["kind"], case.get("k", 1)
    if kind in ("spmv", "spmm", "batch"):
        return {"bytes": 4 * nnz + 8 * n * k, "flops": 2 * nnz * k}
    if kind == "train":  # the words for y, then x and dy in, y, dx and dval out
        return {"bytes": 8 * nnz + 20 * n, "flops": 6 * nnz}
    if kind == "encode":  # CSR in, words out, one product
        return {"bytes": 12 * nnz + 8 * n + 8 * n, "flops": 2 * nnz}
    if kind == "pcg":
        return {"bytes": 16 * nnz + 16 * n, "flops": 4 * nnz}
    if kind == "diff":
        return {"bytes": 20 * nnz + 40 * n, "flops": 8 * nnz}
    return {"bytes": 24 * nnz + 16 * n, "flops": 6 * nnz}


# ---------------------------------------------------------------------------------------------
# 64-bit answers
# ---------------------------------------------------------------------------------------------
def _quantised(case, val):
    """The values that the format stores: binary16, or E8MY (round half away, D + 1 bits cleared)."""
    if case["fmt"] == "fp16":
        return val.to(torch.float16).double()
    d = case["D"]
    bits = val.view(torch.int32)
    sign, mag = bits & -0x80000000, bits & 0x7fffffff
    mag = ((mag + (1 << d)) >> (d + 1)) << (d + 1)
    return (sign | mag).view(torch.float32).double()


def _rows(n, rowptr):
    return torch.repeat_interleave(torch.arange(n, device=DEV), rowptr.diff())


def _product(n, rowptr, col, val, x):
    return torch.zeros((n,) + x.shape[1:], dtype=torch.float64, device=DEV).index_add_(
        0, _rows(n, rowptr), x[col.long()] * (val if x.dim() == 1 else val[:, None]))


def _product_columns(n, rowptr, col, val, x):
    if x.dim() == 1:
        return _product(n, rowptr, col, val, x)
    return torch.cat([_product(n, rowptr, col, val, x[:, j:j + 4].contiguous()) for j in range(0, x.shape[1], 4)], 1)


def _operator(n, rowptr, col, val):
    A = torch.sparse_csr_tensor(rowptr, col.long(), val, size=(n, n))
    row = _rows(n, rowptr)
    d = torch.ones(n, dtype=torch.float64, device=DEV)
    d[row[col == row]] = val[col == row]
    return (lambda v: A @ v), 1.0 / d


def _cg(mul, inv, b, tol, most=20000):
    x, r = torch.zeros_like(b), b.clone()
    z = inv * r
    p, rz, stop = z.clone(), r.dot(z), tol * float(b.norm())
    for it in range(most):
        q = mul(p)
        a = rz / p.dot(q)
        x += a * p
        r -= a * q
        z = inv * r
        new = r.dot(z)
        p = z + (new / rz) * p
        rz = new
        if it % 20 == 19 and float(r.norm()) <= stop:
            break
    return x


def _bicgstab(mul, inv, b, tol, most=4000):
    x, r = torch.zeros_like(b), b.clone()
    hat, p, rho, stop = r.clone(), r.clone(), r.dot(r), tol * float(b.norm())
    for it in range(most):
        ph = inv * p
        v = mul(ph)
        a = rho / hat.dot(v)
        s = r - a * v
        sh = inv * s
        t = mul(sh)
        w = t.dot(s) / t.dot(t)
        x += a * ph + w * sh
        r = s - w * t
        if float(r.norm()) <= stop:
            break
        new = hat.dot(r)
        p = r + (new / rho) * (a / w) * (p - w * v)
        rho = new
    return x


def _solve(n, rowptr, col, val, b, symmetric):
    mul, inv = _operator(n, rowptr, col, val)
    x = torch.zeros_like(b)
    for _ in range(4):  # refined on the true residual
        x = x + (_cg if symmetric else _bicgstab)(mul, inv, b - mul(x), 1e-6)
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind in ("spmv", "spmm", "encode", "train"):
        n, m, rowptr, col, val = _matrix(case, seed)
        q, x = _quantised(case, val), _input(case, m, seed).double()
        if kind == "encode":
            return {"y": _product(n, rowptr, col, q, x), "words": None, "dummies": None, "pad": None}
        if kind == "train":
            dy, row = _uniform(_gen(seed, 7), n).double(), _rows(n, rowptr)
            dx = torch.zeros(m, dtype=torch.float64, device=DEV).index_add_(0, col.long(), q * dy[row])
            return {"y": _product(n, rowptr, col, q, x), "dx": dx, "dval": dy[row] * x[col.long()]}
        y = _product_columns(n, rowptr, col, q, x)
        if case["explicit"]:  # rows by decreasing length inside each sort block, ties in order
            if case["D"] < 15 or case["nx"] * case["ny"] > 1 << 14:
                return None
            at = torch.arange(n, device=DEV)
            key = (at // case["sigma"]) * (1 << 16) + (1 << 15) - rowptr.diff()
            y = y[torch.sort(key, stable=True).indices]
        return y
    if kind == "batch":
        sizes, k = _batch_sizes(case), case["k"]
        rowptr, col, val = _irregular(sizes, seed)
        n = sum(sizes)
        X = _uniform(_gen(seed, 6), n * k).view(n, k).double()
        size = torch.tensor(sizes, device=DEV)
        start = torch.repeat_interleave(torch.cumsum(size, 0) - size, size)
        return _product_columns(n, rowptr, col.long() + start[_rows(n, rowptr)], val.to(torch.float16).double(), X)
    if kind == "pcg":
        n, rowptr, col, val = _poisson7(case, seed)
        return _solve(n, rowptr, col, val, _rhs(n, seed), True)
    if kind == "diff":
        n, rowptr, col, val = _systems(case, seed)
        x = _solve(n, rowptr, col, val, _rhs(n, seed), True)
        lam = _solve(n, rowptr, col, val, _uniform(_gen(seed, 8), n, 0.0, 1.0, torch.float64), True)
        return {"x": x, "dval": -lam[_rows(n, rowptr)] * x[col.long()], "db": lam}
    n, m, rowptr, col, val = _stencil(dict(case, matrix="stencil27"), seed)
    return _solve(n, rowptr, col, _scaled(n, rowptr, col, val), _rhs(n, seed), False)
