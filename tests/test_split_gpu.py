"""SPLIT plans (equal shares of nonzeros per merge thread) against the oracle: nonzero counts at the
edges of a share, a word and a tile, rows that span many tiles, runs of empty rows, ragged and
strided columns, arrays off a 32-byte boundary, values through a permutation, relabelled columns."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

NP = {torch.float64: np.float64, torch.float32: np.float32}
TOL = {torch.float64: 1e-12, torch.float32: 2e-5}
DT = pytest.mark.parametrize("dtype", [torch.float64, torch.float32], ids=["f64", "f32"])


@pytest.fixture(scope="module")
def gbs():
    import paper_1302_1078_gb300 as g

    g.lib()
    return g


def from_lengths(lens, n, seed):
    lens = np.asarray(lens, np.int64)
    rp = np.zeros(lens.size + 1, np.int64)
    np.cumsum(lens, out=rp[1:])
    rng = np.random.default_rng(seed)
    return synth.CSR(lens.size, n, rp.astype(np.int32), rng.integers(0, n, rp[-1]).astype(np.int32),
                     rng.uniform(-1, 1, rp[-1]))


def hubs():
    """Rows of tens of thousands of nonzeros (runs of well over eight tiles) between short and empty ones."""
    rng = np.random.default_rng(3)
    lens = rng.integers(0, 4, 5000)
    lens[[0, 700, 701, 4999]] = [33000, 50001, 4096, 20000]
    lens[1000:3000] = 0
    return from_lengths(lens, 4000, 4)


MATRICES = {f"nnz_{z}": (lambda z=z: from_lengths([0, z - z // 3, 0, z // 3], 50, z))
            for z in (1, 7, 8, 9, 31, 32, 33, 255, 256, 257, 511, 512, 513, 1024, 1025, 4097)}
MATRICES |= {
    "hubs": hubs,
    "singles": lambda: from_lengths(np.ones(3001, int), 3001, 5),
    "stencil2d_37": lambda: synth.stencil2d(37),
    "rmat_13": lambda: synth.rmat(13, ef=16, seed=4),
    "random_rect": lambda: synth.random_csr(333, 1201, 0.02, 5, empty_rows=0.3),
    "dup_unsorted": lambda: synth.random_csr(257, 257, 0.05, 6, sorted_cols=False, duplicates=True),
    "empty_nnz": lambda: synth.random_csr(100, 50, 0.0, 7),
}


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def within(y, ref, r, dtype, what):
    got = y.double().cpu().numpy()
    assert np.all(np.abs(got - ref) <= TOL[dtype] * r), what
    assert np.all(got[r == 0] == 0.0), what


@DT
@pytest.mark.parametrize("name", list(MATRICES))
def test_split_spmv(gbs, name, dtype):
    A = MATRICES[name]()
    v, x = A.vals.astype(NP[dtype]), synth.uniform(A.n, seed=31).astype(NP[dtype])
    ref, r = oracle.spmv(A.m, A.row_ptr, A.col_idx, v, x)
    rp, xd = dev(A.row_ptr), dev(x)
    for off in (0, 1):  # off a 32-byte boundary: element by element
        ci = torch.empty(A.nnz + 8, dtype=torch.int32, device="cuda")[off : off + A.nnz].copy_(dev(A.col_idx))
        vd = torch.empty(A.nnz + 8, dtype=dtype, device="cuda")[off : off + A.nnz].copy_(dev(v))
        plan = gbs.Plan(rp, ci, A.n, dtype, 1)
        for cfg in (dict(), dict(items=8, threads=64), dict(items=8, threads=256)):
            plan.set_config(dict(cfg, variant=6))
            y = plan.spmv(vd, xd, torch.full((A.m,), float("nan"), dtype=dtype, device="cuda"))
            within(y, ref, r, dtype, f"{name} {cfg} off={off}")
            assert torch.equal(y, plan.spmv(vd, xd))
            plan.set_config(dict(cfg, variant=6, relabel=1))
            assert torch.equal(y, plan.spmv(vd, xd)), f"{name} {cfg}: relabelled"


@DT
@pytest.mark.parametrize("k", [1, 2, 3, 5, 8, 16, 33, 70])
@pytest.mark.parametrize("name", ["nnz_1", "nnz_33", "nnz_1025", "hubs", "singles", "rmat_13", "random_rect", "empty_nnz"])
def test_split_spmm(gbs, name, k, dtype):
    A = MATRICES[name]()
    v = A.vals.astype(NP[dtype])
    ld = -(-(k + 1) // 4) * 4  # a row stride above k that keeps rows on 16 bytes
    Xw = synth.uniform(A.n * ld, seed=32, stream=k).reshape(A.n, ld).astype(NP[dtype])
    ref, r = oracle.spmm(A.m, A.row_ptr, A.col_idx, v, Xw[:, :k])
    rp, ci, vd = dev(A.row_ptr), dev(A.col_idx), dev(v)
    plan = gbs.Plan(rp, ci, A.n, dtype, k)
    for items in ((8,) if k == 1 else (32, 64, 256)):
        plan.set_config(dict(variant=6, items=items))
        for X in (dev(Xw[:, :k]), dev(Xw)[:, :k]):
            for Y in (torch.empty((A.m, k), dtype=dtype, device="cuda"),
                      torch.empty((A.m, ld), dtype=dtype, device="cuda")[:, :k]):
                Y.fill_(float("nan"))
                plan.spmm(vd, X, Y)
                within(Y, ref, r, dtype, f"{name} k={k} items={items} ld={X.stride(0)},{Y.stride(0)}")


@DT
@pytest.mark.parametrize("k", [1, 8])
@pytest.mark.parametrize("name", ["nnz_513", "hubs", "rmat_13", "random_rect"])
def test_split_backward(gbs, name, k, dtype):
    """dX = A^T dY with A's values read through the transpose permutation."""
    A = MATRICES[name]()
    v = A.vals.astype(NP[dtype])
    X = synth.uniform(A.n * k, seed=33).reshape(A.n, k).astype(NP[dtype])
    W = synth.uniform(A.m * k, seed=34).reshape(A.m, k).astype(NP[dtype])
    ref, _, r, _ = oracle.backward(A.m, A.n, A.row_ptr, A.col_idx, v, X, W)
    t = gbs.TransposePlan(dev(A.row_ptr), dev(A.col_idx), A.n)
    for items in ((0, 8) if k == 1 else (32, 64)):
        t.set_config(dtype, k, dict(variant=6, items=items))
        assert t.config(dtype, k)["variant"] == 6
        dX, _ = t.backward(dev(v), dev(X[:, 0] if k == 1 else X), dev(W[:, 0] if k == 1 else W))
        within(dX.reshape(A.n, k), ref.reshape(A.n, k), r.reshape(A.n, k), dtype, f"{name} k={k} {items}")


def test_split_is_plans_only(gbs):
    A = MATRICES["singles"]()
    rp, ci, v = dev(A.row_ptr), dev(A.col_idx), dev(A.vals)
    x = torch.zeros(A.n, dtype=torch.float64, device="cuda")
    with pytest.raises(gbs.GbsError):
        gbs.spmv_csr(rp, ci, v, x, config=dict(variant=6))
    plan = gbs.Plan(rp, ci, A.n)
    for bad in (dict(items=7), dict(items=16), dict(threads=512)):
        with pytest.raises(gbs.GbsError):
            plan.set_config(dict(bad, variant=6))


@DT
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 8, 13, 16])
@pytest.mark.parametrize("name", ["nnz_1", "nnz_9", "nnz_257", "hubs", "singles", "rmat_13", "random_rect", "dup_unsorted"])
def test_dvals_from_the_index(gbs, name, k, dtype):
    """dvals with the rows taken from A's index: every width of a gathered slice (32 and 16 bytes, one
    element), column ids on and off a 32-byte boundary."""
    A = MATRICES[name]()
    v = A.vals.astype(NP[dtype])
    for ld in (k, k + 1, -(-k // 4) * 4, -(-k // 8) * 8 + 4):
        Xw = synth.uniform(A.n * ld, seed=35, stream=ld).reshape(A.n, ld).astype(NP[dtype])
        Ww = synth.uniform(A.m * ld, seed=36, stream=ld).reshape(A.m, ld).astype(NP[dtype])
        _, ref, _, r = oracle.backward(A.m, A.n, A.row_ptr, A.col_idx, v, Xw[:, :k].copy(), Ww[:, :k].copy())
        for off in (0, 1):
            ci = torch.empty(A.nnz + 8, dtype=torch.int32, device="cuda")[off : off + A.nnz].copy_(dev(A.col_idx))
            t = gbs.TransposePlan(dev(A.row_ptr), ci, A.n)
            X, W = dev(Xw)[:, :k], dev(Ww)[:, :k]
            _, dvals = t.backward(dev(v), X[:, 0] if k == 1 else X, W[:, 0] if k == 1 else W, need_dX=False)
            within(dvals, ref, r, dtype, f"{name} k={k} ld={ld} off={off}")


@pytest.mark.parametrize("n", [1, 2, 512, 513, 131072, 131073, 262145])
@pytest.mark.parametrize("nnz", [1, 4095, 4096, 4097, 70001])
def test_transpose_tile_and_digit_edges(gbs, nnz, n):
    """The transpose's sort at the edges of its tiles (4096 nonzeros) and digits (9 bits): the stable
    order, the row pointers and the rows, against numpy."""
    rng = np.random.default_rng(nnz + n)
    lens = np.bincount(rng.integers(0, 301, nnz), minlength=301)
    A = from_lengths(lens, n, 6)
    rpT, ciT, perm = (t.cpu().numpy() for t in gbs.TransposePlan(dev(A.row_ptr), dev(A.col_idx), n).arrays())
    order = np.argsort(A.col_idx, kind="stable")
    assert np.array_equal(perm, order)
    assert np.array_equal(ciT, np.repeat(np.arange(A.m), lens)[order])
    assert np.array_equal(rpT, np.concatenate([[0], np.cumsum(np.bincount(A.col_idx, minlength=n))]))


@DT
@pytest.mark.parametrize("nnz", [98303, 98304, 98305])
@pytest.mark.parametrize("shape", ["one_row", "even", "front"])
def test_small_one_shot(gbs, nnz, shape, dtype):
    """The single-launch SpMV at its largest sizes and one past them: every nonzero in one row, even
    rows, and long rows gathered in the first block among short and empty ones."""
    lens = {"one_row": [0, nnz, 0], "even": np.full(nnz // 7 + 1, 7), "front": [nnz // 8] * 5 + [0, 1, 2, 3] * 900}[shape]
    lens = np.asarray(lens, np.int64)
    lens[-1 if shape != "one_row" else 1] += nnz - lens.sum()
    A = from_lengths(lens, 5000, 7)
    v, x = A.vals.astype(NP[dtype]), synth.uniform(A.n, seed=37).astype(NP[dtype])
    ref, r = oracle.spmv(A.m, A.row_ptr, A.col_idx, v, x)
    y = torch.full((A.m,), float("nan"), dtype=dtype, device="cuda")
    gbs.spmv_csr(dev(A.row_ptr), dev(A.col_idx), dev(v), dev(x), y)
    within(y, ref, r, dtype, f"{shape} {nnz}")


@DT
@pytest.mark.parametrize("k", [2, 3, 33, 40, 66, 70])
@pytest.mark.parametrize("name", ["stencil2d_37", "even50", "random_rect"])
def test_rows_tma_tiles_of_both_widths(gbs, name, k, dtype):
    """ROWS_TMA block vectors whose calls have and lack 128-bit column access (different lanes, so
    different row blocks and tiles), several column panels of which the last is narrow, and the
    untuned choice for even rows."""
    A = from_lengths(np.full(1001, 50), 700, 8) if name == "even50" else MATRICES[name]()
    v = A.vals.astype(NP[dtype])
    ld = -(-(k + 1) // 4) * 4
    Xw = synth.uniform(A.n * ld, seed=38, stream=k).reshape(A.n, ld).astype(NP[dtype])
    ref, r = oracle.spmm(A.m, A.row_ptr, A.col_idx, v, Xw[:, :k])
    plan = gbs.Plan(dev(A.row_ptr), dev(A.col_idx), A.n, dtype, k)
    for cfg in (None, dict(variant=3, threads=64), dict(variant=3, threads=256), dict(variant=3, lanes=8, threads=128)):
        if cfg is not None:
            try:
                plan.set_config(cfg)
            except gbs.GbsError as e:
                assert e.status == -8 and cfg["threads"] == 256  # the widest row blocks exceed shared memory
                continue
        for X in (dev(Xw[:, :k]), dev(Xw)[:, :k]):
            within(plan.spmm(dev(v), X), ref, r, dtype, f"{name} k={k} {cfg} ld={X.stride(0)}")


@DT
@pytest.mark.parametrize("length", [5, 20, 27, 50, 52])
@pytest.mark.parametrize("lanes", [2, 4, 8])
def test_rows_tma_row_order_in_a_warp(gbs, lanes, length, dtype):
    """SpMV with half-warps on alternate rows (decided by the row length) and the partial sums' layout:
    every product is the one of ROWS with the same lanes within rounding, and the oracle's."""
    A = from_lengths(np.full(777, length), 900, length)
    v, x = A.vals.astype(NP[dtype]), synth.uniform(A.n, seed=39).astype(NP[dtype])
    ref, r = oracle.spmv(A.m, A.row_ptr, A.col_idx, v, x)
    plan = gbs.Plan(dev(A.row_ptr), dev(A.col_idx), A.n, dtype, 1)
    for threads in (32, 96, 160, 256):
        plan.set_config(dict(variant=3, lanes=lanes, threads=threads))
        within(plan.spmv(dev(v), dev(x)), ref, r, dtype, f"lanes={lanes} threads={threads}")


@pytest.mark.parametrize("k", [1, 8])
def test_capture_of_split_products(gbs, k):
    """A SPLIT plan, a one-shot product (its scratch becomes the graph's) and an untuned backward pass
    captured in one CUDA graph behind an operation that makes their input; replays follow new inputs."""
    A = MATRICES["hubs"]()
    rp, ci, v = dev(A.row_ptr), dev(A.col_idx), dev(A.vals)
    tail = () if k == 1 else (k,)
    x0 = torch.zeros((A.n, *tail), dtype=torch.float64, device="cuda")
    dY = torch.rand((A.m, *tail), dtype=torch.float64, device="cuda")
    plan = gbs.Plan(rp, ci, A.n, torch.float64, k, config=dict(variant=6))
    t = gbs.TransposePlan(rp, ci, A.n)

    def work():
        x = x0 * 2.0
        once = gbs.spmv_csr(rp, ci, v, x) if k == 1 else gbs.spmm_csr(rp, ci, v, x)
        return (plan.spmv(v, x) if k == 1 else plan.spmm(v, x)), once, *t.backward(v, x, dY)

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        work()
    torch.cuda.current_stream().wait_stream(side)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        got = work()
    for seed in (1, 2):
        x0.copy_(dev(synth.uniform(x0.numel(), seed=seed)).reshape(x0.shape))
        g.replay()
        want = work()
        for a, b in zip(got, want):
            assert torch.equal(a, b)


@pytest.mark.parametrize("k", [1, 3, 4])
@pytest.mark.parametrize("m", [5, 20011])
def test_rows_tma_products_in_a_chain(gbs, m, k):
    """Each ROWS_TMA product begins while the one before ends: a chain in which every product reads
    what the last one wrote, behind and before a SPLIT product, with two buffers taken in turn, gives
    the bits of products that are waited for one by one, on a stream and captured."""
    A = from_lengths(np.full(m, 9), m, 9)
    rp, ci, v = dev(A.row_ptr), dev(A.col_idx), dev(A.vals / 3)
    plans = [gbs.Plan(rp, ci, A.n, torch.float64, k, config=dict(variant=q)) for q in (3, 3, 6, 3)]
    x0 = dev(synth.uniform(m * k, seed=41)).reshape((m,) if k == 1 else (m, k))
    bufs = [torch.empty_like(x0), torch.empty_like(x0)]

    def chain(wait):
        x = x0
        for i in range(24):
            p, y = plans[i % 4], bufs[i % 2]
            (p.spmv if k == 1 else p.spmm)(v, x, y)
            x = y
            if wait:
                torch.cuda.synchronize()
        return x

    want = chain(True).clone()
    assert want.abs().max() > 0
    for _ in range(3):
        assert torch.equal(chain(False), want)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = chain(False)
    bufs[0].zero_(), bufs[1].zero_()
    g.replay()
    assert torch.equal(out, want)


@pytest.mark.parametrize("k", [1, 3, 8])
@pytest.mark.parametrize("kept", [dict(variant=1), dict(variant=2), dict(variant=6), dict(variant=6, items=256),
                                  dict(variant=6, relabel=1), dict(variant=3, threads=32)], ids=str)
def test_refused_config_leaves_the_plan_as_it_was(gbs, kept, k):
    """A configuration that is refused, by its arguments or by the row lengths (ROWS_TMA whose row
    blocks do not fit), changes neither the plan's configuration nor its products."""
    A = from_lengths(np.full(40000, 60), 900, 10)
    rp, ci, v = dev(A.row_ptr), dev(A.col_idx), dev(A.vals)
    if k == 1 and "items" in kept:
        kept = dict(kept, items=8)
    plan = gbs.Plan(rp, ci, A.n, torch.float64, k, config=kept)
    X = dev(synth.uniform(A.n * k, seed=42)).reshape((A.n,) if k == 1 else (A.n, k))
    run = plan.spmv if k == 1 else plan.spmm
    config, want = plan.config, run(v, X)
    refused = [dict(variant=6, items=7 if k == 1 else 33), dict(variant=6, items=16 if k == 1 else 512),
               dict(variant=6, items=-32), dict(variant=6, threads=512), dict(variant=2, items=300), dict(variant=99)]
    if k == 1:
        refused.append(dict(variant=3, lanes=1, threads=256))  # row blocks of 15,360 nonzeros
    for bad in refused:
        with pytest.raises(gbs.GbsError):
            plan.set_config(bad)
        assert plan.config == config, bad
        assert torch.equal(run(v, X), want), bad
    plan.set_config(dict(variant=6))
    assert plan.config["variant"] == 6
    plan.set_config(kept)
    assert torch.equal(run(v, X), want)


@DT
def test_odd_block_products_of_one_plan_on_two_streams(gbs, dtype):
    """Block products without 128-bit column access keep their carries to themselves, so one SPLIT
    plan serves several streams at a time: the bits are those of products made one by one."""
    A = synth.rmat(17, ef=16, seed=6)
    rp, ci, v = dev(A.row_ptr), dev(A.col_idx), dev(A.vals.astype(NP[dtype]))
    plan = gbs.Plan(rp, ci, A.n, dtype, 3, config=dict(variant=6))
    X = [dev(synth.uniform(A.n * 3, seed=43, stream=i).astype(NP[dtype])).reshape(A.n, 3) for i in range(2)]
    want = [plan.spmm(v, x).clone() for x in X]
    Y = [[torch.empty_like(want[i]) for _ in range(20)] for i in range(2)]
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    for j in range(20):
        for i in range(2):
            plan.spmm(v, X[i], Y[i][j], stream=streams[i])
    torch.cuda.synchronize()
    for i in range(2):
        assert all(torch.equal(y, want[i]) for y in Y[i])


@pytest.mark.parametrize("k", [1, 4])
@pytest.mark.parametrize("what", ["destroy", "set_config", "graph", "transpose"])
def test_plan_memory_outlives_work_on_another_stream(gbs, what, k):
    """A plan is destroyed or given another configuration, or a transpose plan destroyed, while products
    on a side stream still read what it owns, a graph's replay among them; one-shot products on the
    default stream then draw on the same pool.  Every result is the one of products waited for one by one."""
    A = synth.rmat(17, ef=16, seed=8)
    rp, ci, v = dev(A.row_ptr), dev(A.col_idx), dev(A.vals)
    shape = (A.n,) if k == 1 else (A.n, k)
    X = dev(synth.uniform(A.n * k, seed=44)).reshape(shape)
    once = (lambda: gbs.spmv_csr(rp, ci, v, X)) if k == 1 else (lambda: gbs.spmm_csr(rp, ci, v, X))
    W = dev(synth.uniform(A.m * k, seed=45)).reshape(shape)
    side = torch.cuda.Stream()

    def make():
        if what == "transpose":
            t = gbs.TransposePlan(rp, ci, A.n)
            t.set_config(torch.float64, k, dict(variant=6))
            return t, lambda out, s: out.extend(t.backward(v, X, W, stream=s))
        # (the relabelled ids and x of a graph's ROWS plan stay where they are when its threads change)
        p = gbs.Plan(rp, ci, A.n, torch.float64, k, config=dict(variant=1 if what == "graph" else 6, relabel=1))
        return p, lambda out, s: out.append(p.spmv(v, X, stream=s) if k == 1 else p.spmm(v, X, stream=s))

    plan, go = make()
    want, first = [], once()
    go(want, None)
    for _ in range(5):
        plan, go = make()
        torch.cuda.synchronize()
        got = []
        if what == "graph":
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                for _ in range(20):
                    go(got, None)
            plan.set_config(dict(variant=1, relabel=1, threads=128))
            with torch.cuda.stream(side):
                g.replay()
        else:
            for _ in range(20):
                go(got, side)
        if what == "set_config":
            plan.set_config(dict(variant=4, items=11))
        else:
            del plan, go
        later = [once() for _ in range(10)]
        gbs.lib().gbs_release_scratch()
        torch.cuda.synchronize()
        for i, y in enumerate(got):
            assert torch.equal(y, want[i % len(want)])
        assert all(torch.equal(y, first) for y in later)


def cancelling(m, seed):
    """FP32 rows of up to 41 nonzeros whose products are exact (values +-1, 2 and 4, x of widely
    different size) and whose large terms cancel, at most 256 nonzeros in all (one SPLIT tile, in
    which sums keep both parts)."""
    rng = np.random.default_rng(seed)
    lens = rng.choice([3, 5, 9, 41], m, p=[0.4, 0.4, 0.1, 0.1])
    lens = lens[np.cumsum(lens) <= 256]
    A = from_lengths(lens, 64, seed)
    x = (rng.uniform(0.5, 1, A.n) * 2.0 ** -rng.integers(0, 24, A.n)).astype(np.float32)
    v = rng.choice([1.0, -1.0, 2.0, 4.0], A.nnz).astype(np.float32)
    ci = A.col_idx.copy()
    for i in range(A.m):  # small, large, -large, ...: the pair cancels
        s = A.row_ptr[i]
        ci[s + 1] = ci[s + 2] = int(np.argmax(x))
        ci[s] = int(np.argmin(x))
        v[s + 2] = -v[s + 1]
    return synth.CSR(A.m, A.n, A.row_ptr, ci, v), x


def exact_rows_bound(p):
    """|error| of a compensated sum of the exact terms p (Ogita, Rump and Oishi, 2005): u |sum| +
    (n u)^2 / (1 - n u)^2 * sum |p|, doubled for sums of partial sums."""
    u = 2.0**-24
    g = p.size * u / (1 - p.size * u)
    return 2 * (u * abs(p.sum()) + g * g * np.abs(p).sum())


@pytest.mark.parametrize("route", ["once", "SPLIT k=1", "SPLIT k=3", "SPLIT k=4", "ROWS k=1", "ROWS k=4", "dvals"])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_float_sums_keep_what_cancellation_leaves(gbs, seed, route):
    A, x = cancelling(40, seed)
    rp, ci, v = dev(A.row_ptr), dev(A.col_idx), dev(A.vals)
    if route == "dvals":  # the same sums as dot products over the columns
        k = 41
        X, W = np.zeros((A.m, k), np.float32), np.zeros((A.m, k), np.float32)
        for i in range(A.m):
            s, e = A.row_ptr[i : i + 2]
            X[i, : e - s], W[i, : e - s] = x[A.col_idx[s:e]], A.vals[s:e]
        eye = np.arange(A.m + 1, dtype=np.int32)
        t = gbs.TransposePlan(dev(eye), dev(eye[:-1]), A.m)
        _, got = t.backward(torch.ones(A.m, device="cuda"), dev(X), dev(W), need_dX=False)
        got = got.double().cpu().numpy()[:, None]
    else:
        k = int(route[-1]) if "=" in route else 1
        X = dev(x) if k == 1 else dev(np.repeat(x[:, None], k, 1))
        if route == "once":
            got = gbs.spmv_csr(rp, ci, v, X)
        else:
            plan = gbs.Plan(rp, ci, A.n, torch.float32, k, config=dict(variant=6 if route[0] == "S" else 1))
            got = plan.spmv(v, X) if k == 1 else plan.spmm(v, X)
        got = got.double().cpu().numpy().reshape(A.m, k)
    for i in range(A.m):
        s, e = A.row_ptr[i : i + 2]
        p = A.vals[s:e].astype(np.float64) * x[A.col_idx[s:e]]
        assert np.all(np.abs(got[i] - p.sum()) <= exact_rows_bound(p)), (i, got[i], p)


@pytest.mark.parametrize("k,length", [(1, 131072), (1, 8192), (64, 8192)])
def test_float_hub_rows_round_once(gbs, k, length):
    """FP32 rows of equal signs that span many tiles: the sum is rounded once, the tiles' carries before
    that cost next to nothing (each is rounded, but there are at least 32 of them and their errors average out).  One
    rounding is off by 1/sqrt(12) = 0.289 of the last place in the root mean square; with a fifth more for
    the carries and for the number of rows, 0.35."""
    rows = 8 if k > 1 else 256 if length < 10000 else 48
    A = from_lengths(np.tile([length, 3, 0], rows), 4000, 11)
    rng = np.random.default_rng(12)
    v = rng.uniform(0.5, 1.5, A.nnz).astype(np.float32)
    X = rng.uniform(0.5, 1.5, (A.n, k)).astype(np.float32)
    want = np.zeros((rows, k))
    for i in range(rows):
        s, e = A.row_ptr[3 * i : 3 * i + 2]
        want[i] = v[s:e].astype(np.float64) @ X[A.col_idx[s:e]].astype(np.float64)
    plan = gbs.Plan(dev(A.row_ptr), dev(A.col_idx), A.n, torch.float32, k, config=dict(variant=6))
    got = plan.spmv(dev(v), dev(X[:, 0])) if k == 1 else plan.spmm(dev(v), dev(X))
    got = got.double().cpu().numpy().reshape(A.m, k)[::3]
    err = (got - want) / np.spacing(want.astype(np.float32)).astype(np.float64)
    assert np.sqrt(np.mean(err**2)) <= 0.35


def small_lengths(shape, nnz):
    """Row lengths of at most nnz nonzeros whose long rows lie together, in one cluster's rows."""
    rng = np.random.default_rng(nnz)
    if shape == "block":  # 192 apiece, the rest empty
        lens = np.zeros(max(1, nnz // 192) + 60000, np.int64)
        lens[5 : 5 + nnz // 192] = 192
    elif shape == "just_long":  # just above what a lane or two take by themselves
        lens = np.zeros(70000, np.int64)
        lens[100 : 100 + nnz // 33] = 33
    elif shape == "hub":
        lens = np.zeros(70000, np.int64)
        lens[[69000, 69001, 69002]] = nnz - 6, 5, 1
    elif shape == "few":  # 32 lanes per row
        lens = np.zeros(9, np.int64)
        lens[[0, 3, 8]] = nnz // 2, nnz // 3, nnz // 7
    elif shape == "powers":
        lens = np.minimum(rng.zipf(1.7, 20000), nnz // 10)
        lens[np.cumsum(lens) > nnz] = 0
    return lens


@DT
@pytest.mark.parametrize("nnz", [600, 4097, 32768, 98304])
@pytest.mark.parametrize("shape", ["block", "just_long", "hub", "few", "powers"])
def test_small_one_shot_long_rows_together(gbs, shape, nnz, dtype):
    """The single-launch SpMV whose long rows lie together, on and off a 32-byte boundary: the cluster
    takes their nonzeros in equal parts."""
    A = from_lengths(small_lengths(shape, nnz), 5000, 13)
    v, x = A.vals.astype(NP[dtype]), synth.uniform(A.n, seed=46).astype(NP[dtype])
    ref, r = oracle.spmv(A.m, A.row_ptr, A.col_idx, v, x)
    for off in (0, 1):
        ci = torch.empty(A.nnz + 8, dtype=torch.int32, device="cuda")[off : off + A.nnz].copy_(dev(A.col_idx))
        vd = torch.empty(A.nnz + 8, dtype=dtype, device="cuda")[off : off + A.nnz].copy_(dev(v))
        y = torch.full((A.m,), float("nan"), dtype=dtype, device="cuda")
        gbs.spmv_csr(dev(A.row_ptr), ci, vd, dev(x), y)
        within(y, ref, r, dtype, f"{shape} {nnz} off={off}")
        assert torch.equal(y, gbs.spmv_csr(dev(A.row_ptr), ci, vd, dev(x)))
    rp, xd = dev(A.row_ptr), dev(x)
    with torch.cuda.graph(g := torch.cuda.CUDAGraph()):
        out = gbs.spmv_csr(rp, ci, vd, xd)
    out.zero_()
    g.replay()
    assert torch.equal(out, y)


@pytest.mark.parametrize("shape", ["block", "just_long", "hub"])
def test_small_one_shot_time_does_not_follow_the_row_lengths(gbs, shape):
    """Rows that one after another took forty times merge-path's time do not take twice as long."""
    A = from_lengths(small_lengths(shape, 98304), 60000, 14)
    args = [dev(A.row_ptr), dev(A.col_idx), dev(A.vals), dev(synth.uniform(A.n, seed=47))]
    y = torch.empty(A.m, dtype=torch.float64, device="cuda")

    def us(**kw):
        times = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            for _ in range(20):
                gbs.spmv_csr(*args, y, **kw)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) / 20 * 1e3)
        return min(times)

    assert us() <= 2 * us(config=dict(variant=4, threads=128, items=9))


@DT
@pytest.mark.parametrize("k", [1, 4, 8])
def test_config_of_an_unprepared_transpose(gbs, k, dtype):
    """What a transpose plan reports for a (dtype, k) it has no plan for is what its dX runs: the same
    bits when it is set."""
    A = synth.rmat(14, ef=16, seed=9)
    shape = (A.m,) if k == 1 else (A.m, k)
    W = dev(synth.uniform(A.m * k, seed=49).astype(NP[dtype])).reshape(shape)
    v, X = dev(A.vals.astype(NP[dtype])), torch.zeros_like(W)
    t = gbs.TransposePlan(dev(A.row_ptr), dev(A.col_idx), A.n)
    cfg = t.config(dtype, k)
    assert cfg["variant"] == 6 and cfg["items"] > 0 and cfg["threads"] > 0
    want, _ = t.backward(v, X, W, need_dvals=False)
    t.set_config(dtype, k, cfg)
    assert t.config(dtype, k) == cfg
    assert torch.equal(t.backward(v, X, W, need_dvals=False)[0], want)
    even = synth.stencil2d(37)
    assert gbs.TransposePlan(dev(even.row_ptr), dev(even.col_idx), even.n).config(dtype, k)["variant"] == 1


@pytest.mark.parametrize("scale,ef", [(14, 16), (16, 16), (16, 4)])
def test_untuned_float_vectors_are_as_accurate_as_merge_path(gbs, scale, ef):
    """The default plan of skewed rows, FP32: no further from the exact product than the staged merge-path
    form (a twentieth is what the order of the sums makes on one matrix)."""
    A = synth.rmat(scale, ef=ef, seed=12, vals="u0.5_1.5")
    v, x = A.vals.astype(np.float32), synth.uniform(A.n, seed=51).astype(np.float32)
    ref, _ = oracle.spmv(A.m, A.row_ptr, A.col_idx, v, x)
    rp, ci = dev(A.row_ptr), dev(A.col_idx)

    def error(config):
        y = gbs.Plan(rp, ci, A.n, torch.float32, 1, config=config).spmv(dev(v), dev(x))
        return np.linalg.norm(y.double().cpu().numpy() - ref)

    assert error(None) <= 1.05 * error(dict(variant=2))


def test_release_scratch_gives_memory_back(gbs):
    """What one-shot products leave with the library goes back to the driver, and the next one takes it anew."""
    A = synth.banded(400000, hbw=100, per_row=40, seed=13)
    args = dev(A.row_ptr), dev(A.col_idx), dev(A.vals), dev(synth.uniform(A.n * 4, seed=52)).reshape(A.n, 4)
    want = gbs.spmm_csr(*args)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    gbs.release_scratch()
    assert torch.cuda.mem_get_info()[0] > before
    assert torch.equal(gbs.spmm_csr(*args), want)


@DT
@pytest.mark.parametrize("k,ld", [(2, 2), (3, 3), (3, 4), (5, 5), (4, 4), (7, 8), (8, 8), (12, 12), (13, 13), (13, 16), (16, 16)])
@pytest.mark.parametrize("name", ["rmat_17", "stencil2d_600"])
def test_dvals_of_large_matrices(gbs, name, k, ld, dtype):
    """dvals of matrices whose nonzeros a grid takes in several rounds, rows short and long, in every
    layout of the columns."""
    A = synth.rmat(17, ef=16, seed=14) if name == "rmat_17" else synth.stencil2d(600)
    X = synth.uniform(A.n * ld, seed=53, stream=k).reshape(A.n, ld).astype(NP[dtype])
    W = synth.uniform(A.m * ld, seed=54, stream=k).reshape(A.m, ld).astype(NP[dtype])
    rows = np.repeat(np.arange(A.m), np.diff(A.row_ptr))
    p = W[rows, :k].astype(np.float64) * X[A.col_idx, :k]
    t = gbs.TransposePlan(dev(A.row_ptr), dev(A.col_idx), A.n)
    _, got = t.backward(dev(A.vals.astype(NP[dtype])), dev(X)[:, :k], dev(W)[:, :k], need_dX=False)
    within(got, p.sum(1), np.abs(p).sum(1), dtype, f"{name} k={k} ld={ld}")


@DT
def test_dvals_time_of_odd_columns(gbs, dtype):
    """Thirteen columns in rows of thirteen, which no slice fits, do not take longer than sixteen (by a
    fifth): an X row's lines are used up while they are in L1."""
    A = synth.stencil2d(1000)
    t = gbs.TransposePlan(dev(A.row_ptr), dev(A.col_idx), A.n)
    v = dev(A.vals.astype(NP[dtype]))

    def us(k):
        X, W = (torch.rand((A.n, k), dtype=dtype, device="cuda") for _ in range(2))
        times = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            for _ in range(10):
                t.backward(v, X, W, need_dX=False)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) * 100)
        return min(times)

    assert us(13) <= 1.2 * us(16)


@DT
@pytest.mark.parametrize("k", [1, 4])
def test_backward_beside_itself(gbs, k, dtype):
    """A backward pass whose dvals run beside dX, from the second call on (a transpose used once makes no
    stream): the bits of the two outputs asked for one by one, on two streams and captured before and after."""
    A = synth.rmat(17 if k > 1 or dtype == torch.float32 else 19, ef=16, seed=16)
    shape = (A.m,) if k == 1 else (A.m, k)
    v = dev(A.vals.astype(NP[dtype]))
    X, W = (dev(synth.uniform(A.m * k, seed=55, stream=i).astype(NP[dtype])).reshape(shape) for i in range(2))
    t = gbs.TransposePlan(dev(A.row_ptr), dev(A.col_idx), A.n)
    want = t.backward(v, X, W, need_dvals=False)[0], t.backward(v, X, W, need_dX=False)[1]

    def capture():
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            out = t.backward(v, X, W)
        return g, out

    graphs = [capture(), capture()]  # the second such call is captured: no stream can be made then
    runs = [t.backward(v, X, W) for _ in range(3)]
    graphs.append(capture())
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    runs += [t.backward(v, X, W, stream=side) for _ in range(3)]
    for g, out in graphs:
        out[0].zero_(), out[1].zero_()
        g.replay()
        runs.append(out)
    torch.cuda.synchronize()
    for got in runs:
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


@DT
@pytest.mark.parametrize("k", [3, 5])
def test_tuned_plans_of_odd_columns_serve_padded_operands(gbs, k, dtype):
    """A tuned plan whose columns fill no whole 16 bytes, with contiguous and padded operands, after its
    configuration is set; the padded calls take at most 1.25 times the plan that
    is best for them among the row-wise, merge and split forms (the tuner times cold products, this one warm ones)."""
    A = synth.banded(200000, hbw=500, per_row=41, seed=17)
    v = dev(A.vals.astype(NP[dtype]))
    ld = -(-k // 4) * 4
    Xh = synth.uniform(A.n * ld, seed=56).reshape(A.n, ld).astype(NP[dtype])
    ref, r = oracle.spmm(A.m, A.row_ptr, A.col_idx, A.vals.astype(NP[dtype]), Xh[:, :k])
    X = dev(Xh)
    Y = torch.empty((A.m, ld), dtype=dtype, device="cuda")
    rp, ci = dev(A.row_ptr), dev(A.col_idx)
    plan = gbs.Plan(rp, ci, A.n, dtype, k, tune=True)

    def us(p):
        times = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            for _ in range(10):
                p.spmm(v, X[:, :k], Y[:, :k])
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) * 100)
        return min(times)

    tuned = us(plan)
    within(Y[:, :k], ref, r, dtype, "tuned, padded")
    within(plan.spmm(v, X[:, :k].contiguous()), ref, r, dtype, "tuned, contiguous")
    status = ctypes.c_int(7)
    assert gbs.lib().gbs_plan_status(plan._h, ctypes.byref(status), None) == 0 and status.value == 0
    others = []
    for cfg in (dict(variant=1), dict(variant=2), dict(variant=3, threads=128), dict(variant=5, threads=128), dict(variant=6)):
        plan.set_config(cfg)
        assert plan.config["variant"] == cfg["variant"]
        others.append(us(plan))
        within(Y[:, :k], ref, r, dtype, str(cfg))
    assert tuned <= 1.25 * min(others), (tuned, others)
