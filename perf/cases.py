"""The workloads by which this library's speed is judged, as a program that uses it runs them.

Every case is one call sequence of the public Python interface on one of the matrix families of
the benchmark and the tests: 2D 5-point and 3D 27-point stencils, random banded (FEM-like) rows
and R-MAT graphs, in FP64 and FP32.  A case is a dict:

    op      "once"     one-shot spmv_csr / spmm_csr, nothing kept between calls
            "plan"     a Plan of a fixed structure, multiplied again and again
            "grad"     forward and backward through a CsrOperator
            "gradonce" forward and backward through spmm_autograd (a structure used once)
            "batch"    a BatchedPlan over many uneven matrices
    family  "stencil2d" (size = grid side), "stencil3d" (size = grid side),
            "banded" (size = rows, per_row nonzeros in a band of half-width hbw),
            "rmat" (size = scale, per_row = edge factor)
    dtype   "f64" or "f32";  k: right-hand sides (1: a vector);  tune: the autotuned plan
"""
from __future__ import annotations

import math

import torch

import paper_1302_1078_gb300 as gbs

RMAT_ABCD = (0.57, 0.19, 0.19, 0.05)
DTYPES = {"f64": torch.float64, "f32": torch.float32}
BATCH_KINDS = ("stencil2d", "banded", "rmat")


def _case(name, op, family, size, per_row=0, hbw=0, dtype="f64", k=1, tune=False, count=1):
    return {"name": name, "op": op, "family": family, "size": size, "per_row": per_row, "hbw": hbw, "dtype": dtype,
            "k": k, "tune": tune, "count": count}


def listed():
    return [
        # the smallest call: a 64 x 64 grid Laplacian inside a host-driven loop, where launches and
        # the call's own overhead are what a user waits for
        _case("spmv once lap64", "once", "stencil2d", 64),
        # a structure seen once (an assembled matrix of odd size, single precision, no plan)
        _case("spmv once banded f32", "once", "banded", 200003, 41, 700, "f32"),
        # iterative solvers: the same matrix thousands of times, so the plan is tuned.  The
        # benchmark's three sweep matrices: a regular mesh, FEM-like rows, a power-law graph
        _case("spmv plan 27pt", "plan", "stencil3d", 100, tune=True),
        _case("spmv plan banded", "plan", "banded", 2000000, 50, 1000, tune=True),
        _case("spmv plan rmat22", "plan", "rmat", 22, 16, tune=True),
        # block vectors: four right-hand sides on the mesh without a plan
        _case("spmm once 27pt k4", "once", "stencil3d", 100, k=4),
        # three displacement components in single precision (columns that fill no 128-bit load),
        # plan picked from the row statistics, not tuned
        _case("spmm plan banded k3 f32", "plan", "banded", 500001, 37, 1000, "f32", 3),
        # block vectors on the power-law graph: X (268 MB) is larger than L2
        _case("spmm plan rmat22 k8", "plan", "rmat", 22, 16, k=8, tune=True),
        # training on a fixed graph: Y, dX and dvals each step, a vector in FP64 and features in FP32
        _case("grad rmat20", "grad", "rmat", 20, 16, tune=True),
        _case("grad rmat20 k8 f32", "grad", "rmat", 20, 16, dtype="f32", k=8, tune=True),
        # a sampled subgraph, new every step: statistics, transpose and both passes each time
        _case("gradonce rmat17 k4 f32", "gradonce", "rmat", 17, 16, dtype="f32", k=4),
        # serving: 128 uneven matrices (stencil, banded and R-MAT in turn), eight right-hand sides
        _case("batch 128 k8", "batch", "mixed", 200000, 64, 1000, k=8, tune=True, count=128),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(("once", "once", "plan", "plan", "plan", "grad", "gradonce", "batch"))
    dtype = rng.choice(("f64", "f64", "f32"))
    if op == "batch":
        k = rng.choice((1, 2, 4, 8))
        return {"op": op, "family": "mixed", "size": _log_uniform(rng, 20000, 200000), "per_row": rng.randint(16, 64),
                "hbw": rng.randint(200, 1000), "dtype": dtype, "k": k, "tune": rng.random() < 0.5,
                "count": _log_uniform(rng, 16, 96)}
    family = rng.choice(("stencil2d", "stencil3d", "banded", "banded", "rmat", "rmat"))
    per_row = hbw = 0
    # at most 100 M nonzeros for one product, 16 M for a forward and backward pass, 4 M for a
    # structure used once
    most = {"once": 100_000_000, "plan": 100_000_000, "grad": 16_000_000, "gradonce": 4_000_000}[op]
    if family == "stencil2d":
        size = _log_uniform(rng, 64, min(2048, math.isqrt(most // 5)))
    elif family == "stencil3d":
        size = _log_uniform(rng, 12, min(100, int((most / 27) ** (1 / 3))))
    elif family == "banded":
        per_row, hbw = rng.randint(8, 64), rng.randint(200, 1000)
        size = _log_uniform(rng, 4000, min(2_000_000, most // per_row))
    else:
        per_row = rng.randint(4, 16)
        size = rng.randint(12, min(22, int(math.log2(most / per_row) + 0.07)))
    k = rng.choice((1, 1, rng.randint(2, 16), 4, 8))
    return {"op": op, "family": family, "size": size, "per_row": per_row, "hbw": hbw, "dtype": dtype, "k": k,
            "tune": op in ("plan", "grad") and rng.random() < 0.6, "count": 1}


# ------------------------------------------------------------------ matrices

def _from_mask(mask, cols, vals):
    """CSR of the masked entries of an m x p table of columns and values."""
    m = mask.shape[0]
    row_ptr = torch.zeros(m + 1, dtype=torch.int32, device="cuda")
    row_ptr[1:] = mask.sum(1).cumsum(0)
    return row_ptr, cols[mask].to(torch.int32), vals[mask]


def _stencil2d(N):
    i = torch.arange(N * N, device="cuda", dtype=torch.int32)
    x, y = i % N, i // N
    mask = torch.stack((y > 0, x > 0, x >= 0, x < N - 1, y < N - 1), 1)
    cols = torch.stack((i - N, i - 1, i, i + 1, i + N), 1)
    vals = torch.tensor([-1.0, -1.0, 4.0, -1.0, -1.0], dtype=torch.float64, device="cuda").expand(N * N, 5)
    return (*_from_mask(mask, cols, vals), N * N)


def _stencil3d(N):
    m = N ** 3
    i = torch.arange(m, device="cuda", dtype=torch.int32)
    x, y, z = i % N, i // N % N, i // (N * N)
    d = torch.tensor([(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)], dtype=torch.int32, device="cuda")
    zz, yy, xx = z[:, None] + d[:, 0], y[:, None] + d[:, 1], x[:, None] + d[:, 2]
    mask = (zz >= 0) & (zz < N) & (yy >= 0) & (yy < N) & (xx >= 0) & (xx < N)
    v = torch.full((27,), -1.0, dtype=torch.float64, device="cuda")
    v[13] = 26.0
    return (*_from_mask(mask, (zz * N + yy) * N + xx, v.expand(m, 27)), m)


def _banded(m, per_row, hbw, gen):
    """per_row distinct columns with |i - j| <= hbw in every row, the diagonal among them; N(0,1)
    values and a dominant diagonal."""
    per_row = min(per_row, m)
    cols = torch.empty((m, per_row), dtype=torch.int32, device="cuda")
    vals = torch.randn((m, per_row), dtype=torch.float64, device="cuda", generator=gen)
    off = torch.arange(per_row - 1, device="cuda", dtype=torch.int32)
    for r0 in range(0, m, 500_000):
        r1 = min(m, r0 + 500_000)
        i = torch.arange(r0, r1, device="cuda", dtype=torch.int32)[:, None]
        lo, hi = (i - hbw).clamp_min(0), (i + hbw).clamp_max(m - 1)
        free = hi - lo - (per_row - 2)  # places of a sorted draw with repeats, spread out by `off`
        u = torch.rand((r1 - r0, per_row - 1), device="cuda", generator=gen)
        c = lo + ((u * free).to(torch.int32).minimum(free - 1).sort(1).values + off)
        c += c >= i  # skip the diagonal, which is added
        c = torch.cat((c, i), 1).sort(1).values
        cols[r0:r1] = c
        v = vals[r0:r1]
        v[c == i] = 0
        v[c == i] = v.abs().sum(1) + 1
    row_ptr = torch.arange(0, m * per_row + 1, per_row, dtype=torch.int32, device="cuda")
    return row_ptr, cols.reshape(-1), vals.reshape(-1), m


def _rmat(scale, ef, gen):
    """2^scale vertices, ef * 2^scale generated edges, duplicates removed, values in [0.5, 1.5).  The
    distinct edges are thinned evenly to a count that does not depend on the seed."""
    a, b, c, _ = RMAT_ABCD
    edges = ef << scale
    row = torch.zeros(edges, dtype=torch.int32, device="cuda")
    col = torch.zeros(edges, dtype=torch.int32, device="cuda")
    for _ in range(scale):
        u = torch.rand(edges, device="cuda", generator=gen)
        row.mul_(2).add_(u >= a + b)
        col.mul_(2).add_(((u >= a) & (u < a + b)) | (u >= a + b + c))
    key = torch.unique((row.to(torch.int64) << scale) | col)
    m, nnz = _nnz("rmat", scale, ef)
    assert key.numel() >= nnz
    key = key[torch.arange(nnz, device="cuda") * key.numel() // nnz]
    row_ptr = torch.zeros(m + 1, dtype=torch.int32, device="cuda")
    row_ptr[1:] = torch.bincount(key >> scale, minlength=m).cumsum(0)
    vals = torch.rand(key.numel(), dtype=torch.float64, device="cuda", generator=gen) + 0.5
    return row_ptr, (key & (m - 1)).to(torch.int32), vals, m


def _matrix(family, size, per_row, hbw, gen):
    if family == "stencil2d":
        return _stencil2d(size)
    if family == "stencil3d":
        return _stencil3d(size)
    if family == "banded":
        return _banded(size, per_row, hbw, gen)
    return _rmat(size, per_row, gen)


def _batch_specs(case):
    """(family, size, per_row, hbw) of each member: rows log-uniform up to the case's size, mean row
    length uniform up to its per_row.  They belong to the case, not to the seed."""
    out = []
    for b in range(case["count"]):
        u, v = (b * 0.6180339887498949) % 1.0, (b * 0.7548776662466927 + 0.5) % 1.0
        rows = int(round(1000 * (case["size"] / 1000) ** u))
        avg = 4 + int(v * (case["per_row"] - 3))
        family = BATCH_KINDS[b % 3]
        size = {"stencil2d": max(2, round(math.sqrt(rows))), "banded": rows, "rmat": round(math.log2(rows))}[family]
        out.append((family, size, avg, case["hbw"]))
    return out


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _uniform(shape, dtype, gen):
    return (torch.rand(shape, dtype=torch.float64, device="cuda", generator=gen) * 2 - 1).to(dtype)


def _inputs(case, seed):
    gen, dtype, k = _generator(seed), DTYPES[case["dtype"]], case["k"]
    row_ptr, col_idx, vals, n = _matrix(case["family"], case["size"], case["per_row"], case["hbw"], gen)
    tail = () if k == 1 else (k,)
    X = _uniform((n, *tail), dtype, gen)
    dY = _uniform((n, *tail), dtype, gen) if case["op"] in ("grad", "gradonce") else None
    return row_ptr, col_idx, vals.to(dtype), X, dY


def _batch_inputs(case, seed):
    """The members' matrices, and views of one X and one Y buffer that hold their operands, each
    beginning on a 256-byte boundary."""
    gen, dtype, k = _generator(seed), DTYPES[case["dtype"]], case["k"]
    mats, begin, total = [], [], 0
    for family, size, per_row, hbw in _batch_specs(case):
        rp, ci, v, n = _matrix(family, size, per_row, hbw, gen)
        mats.append((rp, ci, v.to(dtype), n))
        begin.append(total)
        total += -(-n * k // 64) * 64
    X, Y = _uniform((total,), dtype, gen), torch.zeros(total, dtype=dtype, device="cuda")

    def views(buf):
        return [buf[o : o + mat[3] * k].view((mat[3],) if k == 1 else (mat[3], k)) for o, mat in zip(begin, mats)]

    return mats, views(X), views(Y), Y


# ------------------------------------------------------------------- measured

def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        mats, X, Y, out = _batch_inputs(case, seed)
        return {"op": op, "plan": gbs.BatchedPlan(mats, X, Y, tune=case["tune"]), "out": out}
    row_ptr, col_idx, vals, X, dY = _inputs(case, seed)
    state = {"op": op, "k": case["k"], "csr": (row_ptr, col_idx), "vals": vals, "X": X, "dY": dY}
    if op == "plan":
        state["plan"] = gbs.Plan(row_ptr, col_idx, X.shape[0], vals.dtype, case["k"], tune=case["tune"])
    elif op in ("grad", "gradonce"):
        vals.requires_grad_(True)
        X.requires_grad_(True)
        if op == "grad":
            # the operator's plans are made by its first step
            state["op_A"] = gbs.CsrOperator(row_ptr, col_idx, X.shape[0], tune=case["tune"])
            run(state)
    return state


def run(state):
    op = state["op"]
    if op == "batch":
        state["plan"].run()
        return state["out"]
    vals, X = state["vals"], state["X"]
    if op == "once":
        return gbs.spmv_csr(*state["csr"], vals, X) if state["k"] == 1 else gbs.spmm_csr(*state["csr"], vals, X)
    if op == "plan":
        return state["plan"].spmv(vals, X) if state["k"] == 1 else state["plan"].spmm(vals, X)
    Y = state["op_A"](vals, X) if op == "grad" else gbs.spmm_autograd(*state["csr"], vals, X)
    dvals, dX = torch.autograd.grad(Y, (vals, X), state["dY"])
    return {"Y": Y.detach(), "dX": dX, "dvals": dvals}


def _nnz(family, size, per_row):
    """(rows, nonzeros); for R-MAT 2% fewer than the expected number of distinct edges, which every
    seed reaches."""
    if family == "stencil2d":
        return size * size, 5 * size * size - 4 * size
    if family == "stencil3d":
        return size ** 3, (3 * size - 2) ** 3
    if family == "banded":
        return size, size * min(per_row, size)
    a, b, _, d = RMAT_ABCD
    edges, nnz = per_row << size, 0.0
    for i in range(size + 1):  # i levels in quadrant a, l in d, the others in b or c (equal)
        for l in range(size - i + 1):
            j = size - i - l
            cells = math.comb(size, i) * math.comb(size - i, l) * 2 ** j
            nnz += cells * -math.expm1(edges * math.log1p(-(a ** i * d ** l * b ** j)))
    return 1 << size, int(0.98 * nnz)


def work(case):
    es, k = (8 if case["dtype"] == "f64" else 4), case["k"]
    members = _batch_specs(case) if case["op"] == "batch" else [(case["family"], case["size"], case["per_row"], 0)]
    total, flops = 0, 0
    for family, size, per_row, _ in members:
        m, nnz = _nnz(family, size, per_row)
        total += nnz * (4 + es) + 4 * (m + 1) + 2 * m * k * es  # A, X, Y
        flops += 2 * nnz * k
        if case["op"] in ("grad", "gradonce"):
            total += 2 * m * k * es + nnz * es  # dY, dX, dvals
            flops += 4 * nnz * k
    return {"bytes": total, "flops": flops}


# ------------------------------------------------------------------ reference

def _rows(row_ptr, nnz):
    return torch.repeat_interleave(torch.arange(row_ptr.numel() - 1, device="cuda"), row_ptr.diff().long(), output_size=nnz)


def _columns(t):
    return t.double().reshape(t.shape[0], -1)


def _product(m, to, frm, vals, X):
    """sum over the nonzeros of vals * X[frm] into row `to`, in FP64, one column at a time."""
    out = torch.zeros((m, X.shape[1]), dtype=torch.float64, device="cuda")
    for c in range(X.shape[1]):
        out[:, c] = torch.zeros(m, dtype=torch.float64, device="cuda").index_add_(0, to, vals * X[:, c][frm])
    return out


def exact(case, seed):
    if case["op"] == "batch":
        mats, X, _, out = _batch_inputs(case, seed)
        k = case["k"]
        want, o = out.double(), 0
        for (rp, ci, v, n), x in zip(mats, X):
            want[o : o + n * k] = _product(n, _rows(rp, ci.numel()), ci, v.double(), _columns(x)).reshape(-1)
            o += -(-n * k // 64) * 64
        return want
    row_ptr, col_idx, vals, X, dY = _inputs(case, seed)
    rows, v, Xc = _rows(row_ptr, col_idx.numel()), vals.double(), _columns(X)
    Y = _product(X.shape[0], rows, col_idx, v, Xc).reshape(X.shape)
    if dY is None:
        return Y
    dYc = _columns(dY)
    dX = _product(X.shape[0], col_idx, rows, v, dYc).reshape(X.shape)
    dvals = torch.zeros_like(v)
    for c in range(Xc.shape[1]):
        dvals += dYc[:, c][rows] * Xc[:, c][col_idx]
    return {"Y": Y, "dX": dX, "dvals": dvals}
