"""What a user of the library has it do, as cases that can be timed: the products of wide (CSC) and tall (CSR)
sparse matrices with power-law segment lengths and a few very dense segments, alone, in pairs, batched, inside
autograd, inside a least-squares solver, behind the serving runtime and right after ingesting coordinate triples.

``listed()`` gives the fixed cases, ``draw(rng)`` one more of the same ranges, ``prepare`` what a program has in
hand before the call (matrix, vectors, plan), ``run`` one pass through the public entry points, ``work`` the bytes
and operations a pass cannot do without, and ``exact`` the outputs in 64 bits by plain torch.

A case's ``short`` and ``long`` are the indexed and the compressed dimension (rows and columns of a wide matrix,
columns and rows of a tall one), ``nnz`` the nonzeros aimed at, ``empty`` the share of segments without any,
``dense`` the number of very dense segments and ``dense_frac`` their density.
"""
from __future__ import annotations

import math

import torch

import paper_1812_00904_gb300 as pkg

DTYPES = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
VALUE_BYTES = {"f64": 8, "f32": 4, "bf16": 2, "f16": 2}
PLAN_FLAGS = {"stored": 0, "bank": pkg.SPMV_PLAN_BANK_ORDER,
              "rows": pkg.SPMV_PLAN_BANK_ORDER | pkg.SPMV_PLAN_ROW_BLOCKS}

# Vectors per serving request, in turn (requests of 1 to 32 vectors).
REQUEST_VECTORS = (1, 8, 2, 32, 1, 4, 16, 3, 1, 12, 5, 24)


def _case(name, kind, layout, short, long, nnz, dtype="f32", order="stored", exponent=2.0, empty=0.0, dense=0,
          dense_frac=0.0, k=1, count=1):
    c = dict(kind=kind, layout=layout, short=short, long=long, nnz=nnz, dtype=dtype, order=order, exponent=exponent,
             empty=empty, dense=dense, dense_frac=dense_frac, k=k, count=count)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest calls: a model of a few thousand features, one product each way (launch latency)
        _case("tiny_calls_f32", "calls", "csc", 300, 5003, 15_000),
        # the paper's double-precision setting at the size of the small wide workload: one SpMV, one SpVTM
        _case("small_calls_f64", "calls", "csc", 1_000, 100_000, 508_752, "f64", dense=5, dense_frac=0.97),
        # least squares through autograd on the small wide workload with half-size values: forward, d(x), d(values)
        _case("small_grad_bf16", "grad", "csc", 1_000, 100_000, 508_752, "bf16", dense=5, dense_frac=0.97),
        # the same training step on an ordinary document-term matrix, odd sizes and some empty columns
        _case("mid_grad_f16", "grad", "csc", 8_003, 1_000_003, 20_000_000, "f16", empty=0.02, dense=10, dense_frac=0.5),
        # products of a served matrix near the upper end of the serving range of short dimensions
        _case("served_m40k_calls_f32", "calls", "csc", 40_001, 1_500_000, 40_000_000),
        # the document-term workload of the benchmark: a SpMV-SpVTM pair of a wide matrix in bank order
        _case("wide_pair_f32", "pair", "csc", 20_000, 5_000_000, 200_000_000, order="bank", dense=50, dense_frac=0.5),
        # its role-reversed counterpart: a tall matrix, stored order
        _case("tall_pair_f32", "pair", "csr", 2_000, 10_000_000, 150_000_000, exponent=2.2, dense=20, dense_frac=0.6),
        # the product without atomics (bitwise reproducible) over the row-sorted copy
        _case("row_blocks_calls_f32", "calls", "csc", 20_000, 1_250_000, 50_000_000, order="rows", dense=50,
              dense_frac=0.5),
        # eight vectors at once, both ways (block methods, batched inference)
        _case("wide_batch8_f32", "batch", "csc", 20_000, 1_250_000, 50_000_000, dense=50, dense_frac=0.5, k=8),
        # an overdetermined least-squares solve by conjugate gradients in double precision, four iterations
        _case("cgls_f64", "cgls", "csr", 4_000, 400_000, 8_000_000, "f64", dense=5, dense_frac=0.5, k=4),
        # serving: requests of 1 to 32 vectors on eight resident matrices, submitted together
        _case("serve_mixed_f32", "serve", "csc", 1_000, 100_000, 1_000_000, k=24, count=8),
        # ingest of coordinate triples in any order, then one product each way
        _case("ingest_coo_f32", "coo", "csc", 10_007, 500_009, 10_000_000, empty=0.02),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["calls", "calls", "pair", "pair", "grad", "batch", "batch", "cgls", "serve", "coo"])
    layout = rng.choice(["csc", "csr"])
    short = _log(rng, 300, 50_000)
    if kind == "serve":
        return _case("", kind, "csc", 1_000, 100_000, _log(rng, 500_000, 2_000_000), k=rng.randint(8, 24),
                     count=rng.randint(3, 8))
    dtype = {"grad": rng.choice(["bf16", "f16", "f32"]), "batch": "f32",
             "cgls": "f64"}.get(kind, rng.choice(["f32", "f32", "f32", "f64", "bf16", "f16"]))
    if dtype == "f64":
        short = min(short, 12_000)
    most = {"calls": 60e6, "pair": 60e6, "grad": 40e6, "batch": 30e6, "cgls": 20e6, "coo": 20e6}[kind]
    nnz = _log(rng, 15_000 if kind in ("calls", "pair") else 200_000, most)
    # segments of 10 to 120 nonzeros on average, never fuller than a quarter
    long = max(64, int(nnz / min(math.exp(rng.uniform(math.log(10), math.log(120))), short / 4))) | 1
    order = rng.choice(["stored", "bank"]) if kind in ("calls", "pair") else "stored"
    return _case("", kind, layout, short, long, nnz, dtype, order, exponent=rng.choice([2.0, 2.2]),
                 empty=rng.choice([0.0, 0.0, 0.02]), dense=rng.randint(0, 10), dense_frac=0.5,
                 k=rng.choice([2, 4, 8, 16, 32]) if kind == "batch" else rng.randint(2, 4))


# ---------------------------------------------------------------------------
# inputs


def _degrees(short, long, nnz, exponent, empty, dense, dense_frac, gen):
    """Segment lengths of a power law of that density exponent, cut at short, that add up to about nnz."""
    u = 1.0 - torch.rand(long, generator=gen, device="cuda", dtype=torch.float64)
    tail = u ** (-1.0 / (exponent - 1.0))
    keep = torch.rand(long, generator=gen, device="cuda") >= empty
    keep[torch.randint(long, (dense,), generator=gen, device="cuda")] = False
    full = torch.zeros(long, dtype=torch.float64, device="cuda")
    full[torch.randint(long, (dense,), generator=gen, device="cuda")] = max(1.0, dense_frac * short)

    def degrees(d_min):
        d = torch.clamp(torch.floor(d_min * tail), max=0.97 * short) * keep
        return torch.where(full > 0, full, d)

    lo, hi = 1.0, float(short)
    for _ in range(30):
        mid = 0.5 * (lo + hi)
        if float(degrees(mid).sum()) < 1.06 * nnz:
            lo = mid
        else:
            hi = mid
    return degrees(hi)


def _structure(short, long, nnz, exponent, empty, dense, dense_frac, gen):
    """ptr and idx (int32): power-law segment lengths, distinct uniform indices, sorted in every segment; exactly
    nnz nonzeros whatever the seed (the surplus is taken out of segments with several)."""
    deg = _degrees(short, long, nnz, exponent, empty, dense, dense_frac, gen)
    # as many draws as leave that many distinct ones
    draws = torch.round(-short * torch.log1p(-deg / short)).to(torch.int64)
    seg = torch.repeat_interleave(torch.arange(long, device="cuda"), draws)
    key = seg * short + torch.randint(short, (seg.numel(),), generator=gen, device="cuda")
    del seg
    key = torch.sort(key).values
    keep = torch.ones(key.numel(), dtype=torch.bool, device="cuda")
    keep[1:] = key[1:] != key[:-1]
    key = key[keep]
    seg = key // short
    surplus = key.numel() - nnz
    if surplus > 0:
        later = torch.nonzero(seg[1:] == seg[:-1]).flatten() + 1  # not the first of its segment
        # one of every stretch of them, the stretches of equal length
        cut = torch.arange(surplus + 1, device="cuda") * later.numel() // surplus
        at = torch.rand(surplus, generator=gen, device="cuda", dtype=torch.float64) * (cut[1:] - cut[:-1])
        at = torch.minimum(cut[:-1] + at.to(torch.int64), cut[1:] - 1)
        keep = torch.ones(key.numel(), dtype=torch.bool, device="cuda")
        keep[later[at]] = False
        del later, cut, at
        key, seg = key[keep], seg[keep]
    idx = (key - seg * short).to(torch.int32)
    ptr = torch.zeros(long + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(torch.bincount(seg, minlength=long), 0)
    return ptr.to(torch.int32), idx


def _matrix(case, gen):
    ptr, idx = _structure(case["short"], case["long"], case["nnz"], case["exponent"], case["empty"], case["dense"],
                          case["dense_frac"], gen)
    vals = torch.empty(idx.numel(), dtype=torch.float64 if case["dtype"] == "f64" else torch.float32, device="cuda")
    vals = vals.log_normal_(0.0, 1.0, generator=gen).to(DTYPES[case["dtype"]])
    wide = case["layout"] == "csc"
    m, n = (case["short"], case["long"]) if wide else (case["long"], case["short"])
    return dict(layout=case["layout"], m=m, n=n, ptr=ptr, idx=idx, vals=vals)


def _uniform(size, dtype, gen, k=None):
    """U(-1, 1); k vectors lie in rows whose length is a multiple of 16 bytes, as the batched call asks."""
    t = torch.float64 if dtype == "f64" else torch.float32
    shape = size if k is None else (k, -(-size // 4) * 4)
    v = torch.rand(shape, generator=gen, device="cuda", dtype=t).mul_(2.0).sub_(1.0)
    return v if k is None else v[:, :size]


def _served_cases(case):
    """The resident matrices of a serving case: short 1k to 50k, long 100k to 1.6M, nonzeros from the case's up to
    20 times as many, wide and tall in turn (dimensions multiples of 4: packed vectors start on 16 bytes)."""
    out = []
    for i in range(case["count"]):
        f = i / max(1, case["count"] - 1)
        short = 4 * int(1_000 * 50.0 ** ((0.37 * i) % 1.0) / 4)
        long = 4 * int(100_000 * 16.0 ** f / 4)
        out.append(_case("", "calls", "csc" if i % 2 == 0 else "csr", short, long, int(case["nnz"] * 20.0 ** f)))
    return out


def _requests(case):
    """(matrix, op, vectors) of every request of a serving case."""
    return [(r % case["count"], pkg.SPMV_OP_AX if (r // case["count"]) % 2 == 0 else pkg.SPMV_OP_VTA,
             REQUEST_VECTORS[r % len(REQUEST_VECTORS)]) for r in range(case["k"])]


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    kind, dt = case["kind"], case["dtype"]
    if kind == "serve":
        mats = [_matrix(c, gen) for c in _served_cases(case)]
        ins = []
        for i, op, k in _requests(case):
            size = mats[i]["n"] if op == pkg.SPMV_OP_AX else mats[i]["m"]
            ins.append(_uniform(size, dt, gen, k).contiguous())
        return dict(mats=mats, ins=ins)
    A = _matrix(case, gen)
    if kind == "batch":
        return dict(A=A, x=_uniform(A["n"], dt, gen, case["k"]), v=_uniform(A["m"], dt, gen, case["k"]))
    s = dict(A=A, x=_uniform(A["n"], dt, gen), v=_uniform(A["m"], dt, gen))
    if kind == "coo":
        seg = _segments(A)
        order = torch.randperm(seg.numel(), generator=gen, device="cuda")
        major, minor = seg.to(torch.int32)[order], A["idx"][order]
        s["rows"], s["cols"] = (minor, major) if A["layout"] == "csc" else (major, minor)
        s["vals"] = A["vals"][order]
    return s


# ---------------------------------------------------------------------------
# state and one pass


class _Server:
    """A serving runtime with its registered plans; stops with the state."""

    def __init__(self, plans):
        self.plans = plans
        self.handle = pkg.serve_create(64 << 30, k_max=32, n_streams=4)
        self.ids = [pkg.serve_register(self.handle, p.handle) for p in plans]

    def __del__(self):
        if getattr(self, "handle", None):
            pkg.serve_destroy(self.handle)
            self.handle = None


def _plan(A, order="stored"):
    return pkg.Plan(A["m"], A["n"], A["ptr"], A["idx"], A["vals"], layout=A["layout"], flags=PLAN_FLAGS[order])


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    if case["kind"] == "serve":
        s["server"] = _Server([_plan(A) for A in s["mats"]])
        s["requests"] = _requests(case)
        s["outs"] = []
        for i, op, k in s["requests"]:
            A = s["mats"][i]
            s["outs"].append(torch.empty(k, A["m"] if op == pkg.SPMV_OP_AX else A["n"], device="cuda"))
        torch.cuda.synchronize()  # a request's input has to be complete when it is submitted
        return s
    if case["kind"] == "coo":
        return s
    A = s["A"]
    s["plan"] = _plan(A, case["order"])
    if case["kind"] == "grad":
        s["w"] = A["vals"].requires_grad_(True)
        s["x"].requires_grad_(True)
    elif case["kind"] == "batch":
        s["y"] = _padded(case["k"], A["m"], s["x"].dtype)
        s["u"] = _padded(case["k"], A["n"], s["x"].dtype)
    elif case["kind"] == "pair":
        s["y"] = torch.empty(A["m"], dtype=s["x"].dtype, device="cuda")
        s["u"] = torch.empty(A["n"], dtype=s["x"].dtype, device="cuda")
    return s


def _padded(k, size, dtype):
    return torch.empty(k, -(-size // 4) * 4, dtype=dtype, device="cuda")[:, :size]


def run(s):
    kind = s["case"]["kind"]
    if kind == "calls":
        return s["plan"].spmv(s["x"]), s["plan"].spvtm(s["v"])
    if kind == "pair":
        pkg.spmv_pair(s["plan"].handle, s["x"], s["y"], s["v"], s["u"])
        return s["y"], s["u"]
    if kind == "batch":
        s["plan"].batch(pkg.SPMV_OP_AX, s["x"], out=s["y"])
        s["plan"].batch(pkg.SPMV_OP_VTA, s["v"], out=s["u"])
        return s["y"], s["u"]
    if kind == "grad":
        y = pkg.sparse_matvec(s["w"], s["x"], s["plan"])
        loss = 0.5 * (y - s["v"]).square().sum()
        dw, dx = torch.autograd.grad(loss, (s["w"], s["x"]))
        return y.detach(), dw, dx
    if kind == "cgls":
        x, iterations, _ = s["plan"].cgls(s["v"], max_iters=s["case"]["k"], tol=0.0)
        return x, iterations
    if kind == "coo":
        A = s["A"]
        plan = pkg.Plan.from_coo(A["m"], A["n"], s["rows"], s["cols"], s["vals"], layout=A["layout"],
                                 flags=pkg.SPMV_PLAN_COO_UNSORTED)
        y, u = plan.spmv(s["x"]), plan.spvtm(s["v"])
        plan.close()
        return y, u
    server, ids = s["server"], []
    for (i, op, k), xin, out in zip(s["requests"], s["ins"], s["outs"]):
        ids.append(pkg.serve_submit(server.handle, server.ids[i], op, k, xin, out))
    for r in ids:
        pkg.serve_wait(server.handle, r, 60_000)
    return list(s["outs"])


# ---------------------------------------------------------------------------
# what a pass cannot do without


def _product(c, k=1):
    """Bytes and operations of k products of one kind: the matrix read once, the vectors in and out."""
    sv, sx = VALUE_BYTES[c["dtype"]], 8 if c["dtype"] == "f64" else 4
    return c["nnz"] * (4 + sv) + 4 * (c["long"] + 1) + k * sx * (c["short"] + c["long"]), 2 * k * c["nnz"]


def work(case):
    kind = case["kind"]
    sv, sx = VALUE_BYTES[case["dtype"]], 8 if case["dtype"] == "f64" else 4
    if kind == "serve":
        mats = _served_cases(case)
        parts = [_product(mats[i], k) for i, _, k in _requests(case)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    b, f = _product(case, case["k"] if kind == "batch" else 1)
    vectors = sx * (case["short"] + case["long"])
    if kind == "pair":  # one reading of the matrix serves both products
        return {"bytes": b + vectors, "flops": 2 * f}
    if kind == "grad":  # forward; then one reading of indices and values for d(x), d(values) written
        return {"bytes": 2 * b + sv * case["nnz"] + vectors, "flops": 2.5 * f}
    if kind == "cgls":
        return {"bytes": (2 * case["k"] + 2) * b, "flops": (2 * case["k"] + 2) * f}
    if kind == "coo":  # the triples read, the compressed copy written, then the two products
        return {"bytes": case["nnz"] * (12 + 8) + 2 * b, "flops": 2 * f}
    return {"bytes": 2 * b, "flops": 2 * f}


# ---------------------------------------------------------------------------
# the outputs in 64 bits


def _segments(A):
    ptr = A["ptr"].to(torch.int64)
    return torch.repeat_interleave(torch.arange(ptr.numel() - 1, device="cuda"), ptr[1:] - ptr[:-1])


class _Exact:
    def __init__(self, A):
        self.A, self.seg, self.idx = A, _segments(A), A["idx"].to(torch.int64)
        self.a = A["vals"].detach().double()
        self.rows, self.cols = (self.idx, self.seg) if A["layout"] == "csc" else (self.seg, self.idx)

    def ax(self, x):
        y = torch.zeros(self.A["m"], dtype=torch.float64, device="cuda")
        return y.index_add_(0, self.rows, self.a * x.detach().double()[self.cols])

    def vta(self, v):
        u = torch.zeros(self.A["n"], dtype=torch.float64, device="cuda")
        return u.index_add_(0, self.cols, self.a * v.detach().double()[self.rows])


def _exact_cgls(E, b, n, iterations):
    x = torch.zeros(n, dtype=torch.float64, device="cuda")
    r = b.double()
    s = E.vta(r)
    p, gamma = s.clone(), s.dot(s)
    for _ in range(iterations):
        q = E.ax(p)
        alpha = gamma / q.dot(q)
        x = x + alpha * p
        r = r - alpha * q
        s = E.vta(r)
        new = s.dot(s)
        p, gamma = s + (new / gamma) * p, new
    return x


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "serve":
        out = []
        for (i, op, _), xin in zip(_requests(case), s["ins"]):
            E = _Exact(s["mats"][i])
            out.append(torch.stack([E.ax(x) if op == pkg.SPMV_OP_AX else E.vta(x) for x in xin]))
        return out
    E = _Exact(s["A"])
    if kind == "batch":
        return torch.stack([E.ax(x) for x in s["x"]]), torch.stack([E.vta(v) for v in s["v"]])
    if kind == "grad":
        y = E.ax(s["x"])
        r = y - s["v"].double()
        return y, r[E.rows] * s["x"].double()[E.cols], E.vta(r)
    if kind == "cgls":
        return _exact_cgls(E, s["v"], s["A"]["n"], case["k"]), None
    return E.ax(s["x"]), E.vta(s["v"])
