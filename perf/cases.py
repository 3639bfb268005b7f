"""What is timed: the work that programs have this library do, through its
public entry points in ``paper_2112_10037_gb300.api``.

``listed()`` holds the fixed cases, ``draw(rng)`` gives more of the same
ranges.  A case names a ``path`` (which entry point), a ``matrix`` kind with
its sizes, and a value type; ``prepare`` makes the operands on the GPU from
the seed alone, ``run`` is one pass, ``exact`` the same result from plain
torch in 64 bits (expand every product, sort by output entry, add up).  A
case's sizes fix its patterns, the seed its values, so that every seed has
outputs of the same shape.

Matrices (sizes and value ranges as in this repository's generators, made on
the GPU):

* ``lap2d`` / ``lap3d``  5- and 7-point operators on an nx x ny (x nz) grid
  with variable coefficients (diffusion problems),
* ``rmat``               power-law graph adjacency (R-MAT 0.57/0.19/0.19/0.05,
  edge factor ``ef``), cut to its first ``n`` vertices, self-loops dropped,
* ``uniform``            ``lo`` to ``hi`` uniformly random columns per row.
"""
import math

import torch

from paper_2112_10037_gb300 import api

DTYPES = {"f64": torch.float64, "f32": torch.float32}


def listed():
    return [
        # one coarse-grid operator squared: the smallest call a multigrid or
        # smoother set-up makes, where launches and host work are the time
        dict(name="lap2d_64_product", path="product", matrix="lap2d", nx=64, ny=64, dtype="f64"),
        # a full-size PDE operator squared (every row alike and short)
        dict(name="lap3d_96_product", path="product", matrix="lap3d", nx=96, ny=96, nz=96, dtype="f64"),
        # two-hop neighbourhoods of a mid-size graph of odd size, in FP32
        dict(name="rmat_12345_product", path="product", matrix="rmat", n=12345, ef=16, dtype="f32"),
        # two-hop neighbourhoods of a large power-law graph: rows of every
        # length, C three hundred times A (the benchmark's headline workload)
        dict(name="rmat_s18_product", path="product", matrix="rmat", n=262144, ef=16, dtype="f64"),
        # algebraic-multigrid set-up: P^T (A P) from scratch, odd grid
        dict(name="galerkin_61_setup", path="galerkin", nx=61, ny=57, nz=63, agg=2, dtype="f64"),
        # time stepping: the coarse operator again for new values of A, plans
        # kept and both numeric passes in one CUDA graph
        dict(name="galerkin_96_replay", path="galerkin_replay", nx=96, ny=96, nz=96, agg=2, dtype="f64"),
        # many independent products of uneven sizes at once, half stencil
        # squares and half uniformly random operands
        dict(name="batched_64", path="batched", count=64, rows_lo=1024, rows_hi=50000, hi=64, dtype="f64"),
        # a training step through a sparse product with fixed patterns:
        # values of C, then both gradients
        dict(name="train_65536_f32", path="train", matrix="uniform", n=65536, lo=32, hi=32, dtype="f32"),
        dict(name="train_10007_f64", path="train", matrix="uniform", n=10007, lo=2, hi=33, dtype="f64"),
        # triangle counting: (L L) .* L of a graph's strictly lower triangle,
        # edges weighted by their whole-numbered multiplicity (exact sums)
        dict(name="triangles_rmat_s16", path="masked", matrix="rmat", n=65536, ef=16, values="counts", dtype="f64"),
        # CSR to CSC of a large graph, values carried along
        dict(name="transpose_rmat_s20", path="transpose", matrix="rmat", n=1 << 20, ef=16, dtype="f64"),
        # two-hop shortest paths: A (min,+) A
        dict(name="min_plus_rmat_s15", path="semiring", matrix="rmat", n=32768, ef=8, semiring="min_plus",
             dtype="f32"),
    ]


def _log(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, cells):
    """Sides of a box of about `cells` cells whose sides differ by up to 3x."""
    s = cells ** (1.0 / 3.0)
    a, b = rng.uniform(0.6, 1.7), rng.uniform(0.6, 1.7)
    return [max(3, int(s * a)), max(3, int(s * b)), max(3, int(s / (a * b)))]


def draw(rng):
    path = rng.choice(["product", "product", "product", "galerkin", "galerkin_replay", "batched", "train", "masked",
                       "transpose", "semiring"])
    c = dict(path=path, dtype=rng.choice(["f64", "f64", "f32"]))
    if path in ("galerkin", "galerkin_replay"):
        c["nx"], c["ny"], c["nz"] = _grid(rng, _log(rng, 1500, 880000))
        c["agg"] = rng.choice([2, 2, 3])
        return c
    if path == "batched":
        lo = _log(rng, 200, 2000)
        c.update(count=_log(rng, 3, 80), rows_lo=lo, rows_hi=_log(rng, 2 * lo, 40000), hi=rng.randint(8, 64))
        return c
    if path == "train":
        hi = rng.randint(6, 32)
        c.update(matrix="uniform", n=_log(rng, 700, 65000), lo=rng.randint(2, hi), hi=hi)
        return c
    if path == "masked":
        c.update(matrix="rmat", n=_log(rng, 1000, 100000), ef=rng.choice([4, 8, 16]),
                 values=rng.choice(["counts", "uniform"]))
        return c
    c["matrix"] = rng.choice(["lap2d", "lap3d", "rmat", "rmat", "uniform"])
    if c["matrix"] == "lap2d":
        cells = _log(rng, 1000, 1500000)
        c["nx"] = max(3, int(math.sqrt(cells) * rng.uniform(0.4, 2.0)))
        c["ny"] = max(3, cells // c["nx"])
    elif c["matrix"] == "lap3d":
        c["nx"], c["ny"], c["nz"] = _grid(rng, _log(rng, 1000, 880000))
    elif c["matrix"] == "rmat":
        c.update(n=_log(rng, 1000, 800000 if path == "transpose" else 150000), ef=rng.choice([4, 8, 16]))
    else:
        hi = rng.randint(6, 64)
        c.update(n=_log(rng, 700, 50000), lo=rng.randint(2, hi), hi=hi)
    if path == "semiring":
        c["semiring"] = rng.choice(["min_plus", "min_plus", "max_plus", "or_and"])
    return c


# ------------------------------------------------------------------ matrices

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed):
    return torch.Generator(device=_device()).manual_seed(int(seed) * 7919 + 11)


def _pattern_gen(*sizes):
    """Generator of a pattern: the same for every seed."""
    h = 1
    for x in sizes:
        h = (h * 1000003 + int(x)) % (1 << 40)
    return torch.Generator(device=_device()).manual_seed(h)


def _csr(nrows, ncols, key, vals, dtype):
    """CSR from ascending distinct keys row * ncols + column."""
    rows = torch.div(key, ncols, rounding_mode="floor")
    rp = torch.zeros(nrows + 1, dtype=torch.int32, device=key.device)
    rp[1:] = torch.cumsum(torch.bincount(rows, minlength=nrows), 0)
    return api.DeviceCSR(nrows, ncols, rp, (key - rows * ncols).to(torch.int32), vals.to(dtype))


def _stencil(dims, g, dtype):
    """5- or 7-point operator on a box, x fastest; off-diagonal -U(0.5, 1.5),
    diagonal twice the number of axes times U(0.5, 1.5)."""
    dev = _device()
    n = math.prod(dims)
    cell = torch.arange(n, device=dev)
    keys, stride = [cell * n + cell], 1
    for d in dims:
        x = torch.div(cell, stride, rounding_mode="floor") % d
        down, up = cell[x > 0], cell[x < d - 1]
        keys += [down * n + down - stride, up * n + up + stride]
        stride *= d
    key = torch.sort(torch.cat(keys)).values
    v = torch.rand(key.numel(), generator=g, device=dev, dtype=torch.float64) + 0.5
    on_diagonal = torch.div(key, n, rounding_mode="floor") == key % n
    return _csr(n, n, key, torch.where(on_diagonal, 2.0 * len(dims) * v, -v), dtype)


def _rmat(n, ef, g, dtype):
    dev, gp = _device(), _pattern_gen(n, ef)
    scale = max(1, (n - 1).bit_length())
    e = int(ef * n)
    row = torch.zeros(e, dtype=torch.int64, device=dev)
    col = torch.zeros(e, dtype=torch.int64, device=dev)
    for _ in range(scale):
        u = torch.rand(e, generator=gp, device=dev)
        row = 2 * row + (u >= 0.76)
        col = 2 * col + (((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
    keep = (row != col) & (row < n) & (col < n)
    key = torch.unique(row[keep] * n + col[keep])
    return _csr(n, n, key, torch.rand(key.numel(), generator=g, device=dev, dtype=torch.float64) + 0.5, dtype)


def _uniform(n, ncols, lo, hi, g, dtype, which=0):
    """lo to hi uniformly random columns per row (repeats merged), N(0,1)."""
    dev, gp = _device(), _pattern_gen(n, ncols, lo, hi, which)
    counts = torch.randint(lo, hi + 1, (n,), generator=gp, device=dev)
    rows = torch.repeat_interleave(torch.arange(n, device=dev), counts)
    cols = torch.randint(0, ncols, (rows.numel(),), generator=gp, device=dev)
    key = torch.unique(rows * ncols + cols)
    return _csr(n, ncols, key, torch.randn(key.numel(), generator=g, device=dev, dtype=torch.float64), dtype)


def _matrix(case, g, which=0):
    dt, kind = DTYPES[case["dtype"]], case["matrix"]
    if kind == "lap2d":
        return _stencil((case["nx"], case["ny"]), g, dt)
    if kind == "lap3d":
        return _stencil((case["nx"], case["ny"], case["nz"]), g, dt)
    if kind == "rmat":
        return _rmat(case["n"], case["ef"], g, dt)
    return _uniform(case["n"], case["n"], case["lo"], case["hi"], g, dt, which)


def _aggregation(case, g, dtype):
    """P: each fine cell belongs to one agg^3 aggregate, weight U(0.5, 1.5)."""
    nx, ny, nz, a = case["nx"], case["ny"], case["nz"], case["agg"]
    cx, cy, cz = -(-nx // a), -(-ny // a), -(-nz // a)
    i = torch.arange(nx * ny * nz, device=_device())
    x, y, z = i % nx, torch.div(i, nx, rounding_mode="floor") % ny, torch.div(i, nx * ny, rounding_mode="floor")
    x, y, z = (torch.div(t, a, rounding_mode="floor") for t in (x, y, z))
    v = torch.rand(i.numel(), generator=g, device=i.device, dtype=torch.float64) + 0.5
    return _csr(i.numel(), cx * cy * cz, i * (cx * cy * cz) + (z * cy + y) * cx + x, v, dtype)


def _batch_shapes(case):
    """(kind, rows) of every instance: rows log-spaced over the range, kinds
    in turn."""
    n, lo, hi = case["count"], case["rows_lo"], case["rows_hi"]
    kinds = ("lap2d", "uniform", "lap3d", "uniform")
    return [(kinds[i % 4], int(lo * (hi / lo) ** ((i + 0.5) / n))) for i in range(n)]


def _batch_pairs(case, g):
    dt, pairs = DTYPES[case["dtype"]], []
    for kind, r in _batch_shapes(case):
        if kind == "uniform":
            pairs.append(tuple(_uniform(r, r, 2, case["hi"], g, dt, which) for which in (0, 1)))
        else:
            d = 2 if kind == "lap2d" else 3
            A = _stencil((max(3, round(r ** (1.0 / d))),) * d, g, dt)
            pairs.append((A, A))
    return pairs


def _operands(case, seed):
    """The operands of the case's product(s), as DeviceCSR."""
    g = _gen(seed)
    path = case["path"]
    if path in ("galerkin", "galerkin_replay"):
        A = _stencil((case["nx"], case["ny"], case["nz"]), g, DTYPES[case["dtype"]])
        return _aggregation(case, g, DTYPES[case["dtype"]]), A
    if path == "batched":
        return _batch_pairs(case, g)
    A = _matrix(case, g)
    if path == "masked":
        # strictly lower triangle of the undirected simple graph
        r = torch.repeat_interleave(torch.arange(A.nrows, device=A.col_idx.device), A.row_ptr.diff().long())
        c = A.col_idx.long()
        key = torch.unique(torch.maximum(r, c) * A.ncols + torch.minimum(r, c))
        v = torch.rand(key.numel(), generator=g, device=key.device, dtype=torch.float64) + 0.5
        if case["values"] == "counts":
            v = torch.ceil(2 * v)  # 1, 2 or 3 parallel edges
        L = _csr(A.nrows, A.ncols, key, v, DTYPES[case["dtype"]])
        return L, L
    if case.get("matrix") == "uniform" and path != "transpose":
        return A, _matrix(case, g, 1)  # two independent operands
    return A, A


# ------------------------------------------------------------ prepare and run

def prepare(case, seed):
    path, dt = case["path"], DTYPES[case["dtype"]]
    ops = _operands(case, seed)
    if path == "batched":
        return dict(path=path, pairs=ops, dtype=dt)
    state = dict(path=path, A=ops[0], B=ops[1], dtype=dt, semiring=case.get("semiring"))
    if path == "train":  # patterns are fixed for the whole training run
        op = api.SparseMatmul(ops[0], ops[1], dtype=dt)
        w = torch.randn(op.nnz, generator=_gen(seed + 1), device=ops[0].vals.device, dtype=dt)
        state.update(op=op, w=w, a=ops[0].vals.clone().requires_grad_(), b=ops[1].vals.clone().requires_grad_())
    elif path == "galerkin_replay":
        state["chain"] = api.Galerkin(ops[0], ops[1], dtype=dt)
        state["chain"].capture()
    return state


def _parts(C):
    return {"row_ptr": C.row_ptr, "col_idx": C.col_idx, "vals": C.vals}


def run(s):
    path = s["path"]
    if path == "product":
        return _parts(api.spgemm(s["A"], s["B"], dtype=s["dtype"]))
    if path == "semiring":
        return _parts(api.spgemm_semiring(s["A"], s["B"], semiring=s["semiring"], dtype=s["dtype"]))
    if path == "galerkin":
        return _parts(api.galerkin(s["A"], s["B"], dtype=s["dtype"]))
    if path == "galerkin_replay":
        return _parts(s["chain"].replay())
    if path == "batched":
        b = api.Batch(s["pairs"], dtype=s["dtype"])
        b.symbolic()
        b.numeric()
        return [_parts(w) for w in b.waves]  # each wave's products, stacked
    if path == "train":
        c = s["op"](s["a"], s["b"])
        da, db = torch.autograd.grad(c, (s["a"], s["b"]), s["w"])
        return {"c": c, "da": da, "db": db}
    if path == "masked":
        return api.masked_spgemm(s["A"], s["B"], s["A"], dtype=s["dtype"])
    return _parts(api.transpose(s["A"]))


# ---------------------------------------------------------------- references

CHUNK = 100_000_000  # products expanded at a time


def _rows_of(M):
    return torch.repeat_interleave(torch.arange(M.nrows, device=M.col_idx.device), M.row_ptr.diff().long())


def _product_counts(A, B):
    """Products of every nonzero of A (the length of its row of B)."""
    return B.row_ptr.diff().long()[A.col_idx.long()]


def _expand(A, B, e0, e1, counts):
    """Every product of A's nonzeros [e0, e1): (position in A, position in B)."""
    c = counts[e0:e1]
    e = torch.repeat_interleave(torch.arange(e0, e1, device=c.device), c)
    first = torch.cumsum(c, 0) - c
    q = torch.arange(e.numel(), device=c.device) - first[e - e0] + B.row_ptr.long()[A.col_idx.long()[e]]
    return e, q


def _row_chunks(A, counts):
    """Row ranges of about CHUNK products, as (first row, last row)."""
    per_nnz = torch.cat([counts.new_zeros(1), torch.cumsum(counts, 0)])
    total = per_nnz[A.row_ptr.long()].cpu()
    r = 0
    while r < A.nrows:
        t = int(torch.searchsorted(total, total[r] + CHUNK, right=True)) - 1
        t = min(max(t, r + 1), A.nrows)
        yield r, t
        r = t


def _reduce(a, b, where, n, semiring):
    if semiring in (None, "plus_times"):
        return torch.zeros(n, dtype=torch.float64, device=a.device).index_add_(0, where, a * b)
    if semiring == "or_and":
        return torch.zeros(n, dtype=torch.float64, device=a.device).index_reduce_(
            0, where, ((a != 0) & (b != 0)).double(), "amax")
    zero = math.inf if semiring == "min_plus" else -math.inf
    return torch.full((n,), zero, dtype=torch.float64, device=a.device).index_reduce_(
        0, where, a + b, "amin" if semiring == "min_plus" else "amax")


def _exact_product(A, B, semiring=None):
    counts = _product_counts(A, B)
    rows, rp = _rows_of(A), A.row_ptr.long()
    av, bv, bc = A.vals.double(), B.vals.double(), B.col_idx.long()
    keys, vals = [], []
    for r0, r1 in _row_chunks(A, counts):
        e, q = _expand(A, B, int(rp[r0]), int(rp[r1]), counts)
        key, where = torch.unique((rows[e] - r0) * B.ncols + bc[q], return_inverse=True)
        vals.append(_reduce(av[e], bv[q], where, key.numel(), semiring))
        keys.append((key + r0 * B.ncols) if key.numel() else key)
        del e, q, where
    key = torch.cat(keys) if keys else torch.zeros(0, dtype=torch.int64, device=av.device)
    del keys
    return _csr(A.nrows, B.ncols, key, torch.cat(vals) if vals else av[:0], torch.float64)


def _exact_transpose(M):
    key = M.col_idx.long() * M.nrows + _rows_of(M)
    order = torch.argsort(key)
    return _csr(M.ncols, M.nrows, key[order], M.vals.double()[order], torch.float64)


def exact(case, seed):
    path = case["path"]
    ops = _operands(case, seed)
    if path in ("product", "semiring"):
        return _parts(_exact_product(*ops, semiring=case.get("semiring")))
    if path in ("galerkin", "galerkin_replay"):
        return _parts(_exact_product(_exact_transpose(ops[0]), _exact_product(ops[1], ops[0])))
    if path == "transpose":
        return _parts(_exact_transpose(ops[0]))
    if path == "batched":
        got = [_exact_product(a, b) for a, b in ops]
        base = [0]
        for c in got:
            base.append(base[-1] + c.nnz)
        rp = torch.cat([c.row_ptr[:-1] + o for c, o in zip(got, base)] + [got[-1].row_ptr[-1:] + base[-2]])
        return [{"row_ptr": rp, "col_idx": torch.cat([c.col_idx for c in got]),
                 "vals": torch.cat([c.vals for c in got])}]
    A, B = ops
    counts = _product_counts(A, B)
    av, bv = A.vals.double(), B.vals.double()
    rows, rp = _rows_of(A), A.row_ptr.long()
    if path == "masked":
        mkey = rows * A.ncols + A.col_idx.long()
        out = torch.zeros(A.nnz, dtype=torch.float64, device=av.device)
        for r0, r1 in _row_chunks(A, counts):
            e, q = _expand(A, B, int(rp[r0]), int(rp[r1]), counts)
            key = rows[e] * A.ncols + B.col_idx.long()[q]
            at = torch.searchsorted(mkey, key).clamp_(max=A.nnz - 1)
            hit = mkey[at] == key
            out.index_add_(0, at[hit], av[e[hit]] * bv[q[hit]])
        return out * av
    C = _exact_product(A, B)
    dt = DTYPES[case["dtype"]]
    w = torch.randn(C.nnz, generator=_gen(seed + 1), device=av.device, dtype=dt).double()
    ckey = _rows_of(C) * C.ncols + C.col_idx.long()
    da, db = torch.zeros_like(av), torch.zeros_like(bv)
    for r0, r1 in _row_chunks(A, counts):
        e, q = _expand(A, B, int(rp[r0]), int(rp[r1]), counts)
        dc = w[torch.searchsorted(ckey, rows[e] * C.ncols + B.col_idx.long()[q])]
        da.index_add_(0, e, dc * bv[q])
        db.index_add_(0, q, av[e] * dc)
    return {"c": C.vals, "da": da, "db": db}


# ------------------------------------------------------------ cost, tolerance

def _sizes(A, B):
    """(products, entries of C); C's entries counted on every s-th row of A
    where the product is large, and scaled by the products."""
    counts = _product_counts(A, B)
    total = int(counts.sum())
    s = 1 + total // 200_000_000
    rows, rp = _rows_of(A), A.row_ptr.long()
    seen, distinct = 0, 0
    for r0, r1 in _row_chunks(A, counts):
        e0, e1 = int(rp[r0]), int(rp[r1])
        c = torch.where(rows[e0:e1] % s == 0, counts[e0:e1], 0)
        e, q = _expand(A, B, e0, e1, torch.cat([counts.new_zeros(e0), c]))
        seen += e.numel()
        distinct += int(torch.unique((rows[e] - r0) * B.ncols + B.col_idx.long()[q]).numel())
    return total, int(distinct * (total / max(seen, 1)))


def work(case):
    """Each operand read once, each result written once (row pointers and
    columns 4 bytes, values 4 or 8), and two operations per product.  For a
    fixed pattern (train, replay) C's structure is read or written as the
    entry point does: its numeric pass writes C's columns with its values."""
    path = case["path"]
    vb = 8 if case["dtype"] == "f64" else 4
    ops = _operands(case, 0)

    def size(M):
        return 4 * (M.nrows + 1) + (4 + vb) * M.nnz

    if path == "batched":
        read = sum(size(A) + (0 if A is B else size(B)) for A, B in ops)
        both = [_sizes(A, B) for A, B in ops]
        return {"bytes": read + sum(4 * (A.nrows + 1) + (4 + vb) * c for (A, _), (_, c) in zip(ops, both)),
                "flops": 2 * sum(p for p, _ in both)}
    A, B = ops
    if path in ("galerkin", "galerkin_replay"):
        P, A = ops
        AP = _exact_product(A, P)
        R = _exact_transpose(P)
        p2, c2 = _sizes(R, AP)
        # A, P and the coarse operator; A P is an intermediate result
        return {"bytes": size(A) + size(P) + 4 * (P.ncols + 1) + (4 + vb) * c2,
                "flops": 2 * (int(_product_counts(A, P).sum()) + p2)}
    if path == "transpose":
        return {"bytes": size(A) + 4 * (A.ncols + 1) + (4 + vb) * A.nnz, "flops": 0}
    if path == "masked":  # the graph once, one value per entry of the mask
        return {"bytes": size(A) + vb * A.nnz, "flops": 2 * int(_product_counts(A, B).sum())}
    products, nnz = _sizes(A, B)
    read = size(A) + (0 if A is B else size(B))
    if path == "train":  # forward, then dC read once and both gradients written
        return {"bytes": read + (4 + vb) * nnz + (4 + vb) * nnz + vb * (A.nnz + B.nnz), "flops": 6 * products}
    return {"bytes": read + 4 * (A.nrows + 1) + (4 + vb) * nnz, "flops": 2 * products}


def tolerance(case):
    """Sums in another order at the same precision; structure, moved values
    and exact sums (counts, min, max, or) stay the same."""
    path = case["path"]
    if path in ("transpose", "semiring") or (path == "masked" and case["values"] == "counts"):
        return "exact"
    if case["dtype"] == "f64":
        return {"rel": 3e-15, "max": 1e-14}
    return {"rel": 5e-7, "max": 5e-6}
