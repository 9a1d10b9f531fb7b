"""The one-vector passes of validated plans (pass_kernel.cuh): products against the FP64 oracle,
dot products bit for bit against the streaming kernel (an unvalidated plan of the same tiles),
at the edges of steps and tiles, with empty segments anywhere, and from many copies of a short
accumulator to the longest one that fits in shared memory."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import synth  # noqa: E402

import paper_1812_00904_gb300 as pkg  # noqa: E402
from gpu_util import DEV, TOL, assert_close, check_products, dev_vec, host_of, make_plan  # noqa: E402

DTYPES = [torch.float64, torch.float32, torch.bfloat16, torch.float16]


def _degrees(kind, nnz, rng, short):
    if kind == "one":  # one long segment (repeated indices), empty ones before and after
        return np.array([0, 0, nnz, 0])
    if kind == "single":  # a head at every position
        return np.ones(nnz, dtype=np.int64)
    deg = []  # segments of 0 to 90 nonzeros, empty ones at both ends and in runs
    left = nnz
    deg += [0, 0, 0]
    while left > 0:
        d = int(min(left, rng.integers(0, 90) if rng.random() < 0.7 else rng.integers(0, 4)))
        deg.append(d)
        if rng.random() < 0.02:
            deg += [0] * int(rng.integers(1, 40))
        left -= d
    return np.array(deg + [0, 0])


def _check(A, dtype, tile_items, what):
    plan, stored = make_plan(A, dtype, tile_items=tile_items)
    x, v = synth.uniform_vector(A.n, 3), synth.uniform_vector(A.m, 4)
    check_products(plan, stored, x, v, TOL[dtype], what)
    ref, _ = make_plan(A, dtype, tile_items=tile_items, flags=pkg.SPMV_PLAN_NO_VALIDATE)
    xd, vd = dev_vec(x, plan.vec_dtype), dev_vec(v, plan.vec_dtype)
    dot = (lambda p: p.spvtm(vd)) if A.layout == "csc" else (lambda p: p.spmv(xd))
    assert torch.equal(dot(plan), dot(ref)), f"{what}: dot products differ from the streaming kernel's"
    y, u = torch.full((A.m,), 7.0, dtype=plan.vec_dtype, device=DEV), torch.full((A.n,), 7.0, dtype=plan.vec_dtype, device=DEV)
    pkg.spmv_pair(plan.handle, xd, y, vd, u)
    assert torch.equal(u if A.layout == "csc" else y, dot(plan)), f"{what}: the pair's dot products differ"
    short, ref_s, scale = ((y, oracle.spmv, oracle.abs_spmv) if A.layout == "csc" else (u, oracle.spvtm, oracle.abs_spvtm))
    arg = host_of(xd if A.layout == "csc" else vd)
    assert_close(host_of(short), ref_s(stored, arg), scale(stored, arg), TOL[dtype], f"{what}: pair")
    r, z = dev_vec(synth.uniform_vector(A.m, 5), plan.vec_dtype), dev_vec(synth.uniform_vector(A.n, 6), plan.vec_dtype)
    g = plan.dvalues(r, z)
    assert torch.equal(g, ref.dvalues(r, z)), f"{what}: the values' gradient differs from the streaming kernel's"
    exact = oracle.dvalues(stored, host_of(r), host_of(z))
    unit = {torch.bfloat16: 2.0**-8, torch.float16: 2.0**-11}.get(dtype, 2.0**-23)
    assert np.all(np.abs(host_of(g) - exact) <= unit * np.abs(exact) + 2.0**-24), f"{what}: dvalues"
    plan.check()


@pytest.mark.parametrize("dtype", DTYPES, ids=str)
@pytest.mark.parametrize("layout", ["csc", "csr"])
@pytest.mark.parametrize("kind", ["one", "single", "mixed"])
def test_edges_of_steps_and_tiles(kind, layout, dtype):
    rng = np.random.default_rng(5)
    for tile_items in (256, 512, 768):
        for nnz in (1, 8, 255, 256, 257, 511, 513, 769, 60_000):
            deg = _degrees(kind, nnz, rng, 300)
            m, n = (300, len(deg)) if layout == "csc" else (len(deg), 300)
            A = synth.random_matrix(m, n, layout, degrees=deg, seed=nnz, duplicates=True)
            _check(A, dtype, tile_items, f"{kind} {layout} nnz={nnz} T={tile_items}")


@pytest.mark.parametrize("dtype", DTYPES, ids=str)
@pytest.mark.parametrize("short", [1, 31, 4000, 14_000, 23_000, 27_000, 48_000, 52_001, 57_000])
def test_length_of_the_short_vector(short, dtype):
    # from 16 copies of the accumulator to one beside the staging of a few warps, and beyond
    rng = np.random.default_rng(short)
    deg = np.minimum((3.0 * rng.random(20_000) ** -1.0).astype(np.int64), 3_000)
    A = synth.random_matrix(short, 20_000, "csc", degrees=deg, seed=9, duplicates=True)
    _check(A, dtype, 256, f"short={short}")


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32, torch.bfloat16], ids=str)
@pytest.mark.parametrize("short,nnz", [(513, 200), (9_451, 2_000), (22_000, 30_000), (45_889, 26_428)])
def test_few_tiles_beside_a_long_short_vector(short, nnz, dtype):
    """More warps move the short vectors than there are tiles to work on."""
    rng = np.random.default_rng(short)
    deg = np.minimum(rng.integers(1, 2_000, 300), short)
    deg = deg[: np.searchsorted(np.cumsum(deg), nnz) + 1]
    for layout, m, n in (("csc", short, len(deg)), ("csr", len(deg), short)):
        _check(synth.random_matrix(m, n, layout, degrees=deg, seed=5, duplicates=True), dtype, 256, f"{layout} {short}")


def test_in_a_graph_and_with_changed_values():
    """A captured pair replays on new vectors and on values changed in place (the plan borrows them)."""
    rng = np.random.default_rng(8)
    A = synth.random_matrix(2_000, 30_000, "csc", degrees=rng.integers(0, 40, 30_000), seed=2)
    plan, stored = make_plan(A)
    xd, vd = dev_vec(synth.uniform_vector(A.n, 1), torch.float32), dev_vec(synth.uniform_vector(A.m, 2), torch.float32)
    y, u = torch.empty(A.m, device=DEV), torch.empty(A.n, device=DEV)
    pkg.spmv_pair(plan.handle, xd, y, vd, u)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        pkg.spmv_pair(plan.handle, xd, y, vd, u)
    plan.vals.mul_(-2.0)
    xd.mul_(3.0)
    g.replay()
    torch.cuda.synchronize()
    stored = synth.SparseMatrix(A.layout, A.m, A.n, A.ptr, A.idx, -2.0 * stored.vals)
    xs, vs = host_of(xd), host_of(vd)
    assert_close(host_of(y), oracle.spmv(stored, xs), oracle.abs_spmv(stored, xs), 1e-5, "y")
    assert_close(host_of(u), oracle.spvtm(stored, vs), oracle.abs_spvtm(stored, vs), 1e-5, "u")


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float16], ids=str)
@pytest.mark.parametrize("layout", ["csc", "csr"])
@pytest.mark.parametrize("short", [4, 300, 5_000, 9_000, 20_000, 56_000])
def test_several_vectors(short, layout, dtype):
    """Batches of either direction against the oracle, on and off chip; the dot products equal the
    single ones bit for bit."""
    rng = np.random.default_rng(short)
    for k, nnz in ((2, 256), (3, 257), (4, 30_011), (5, 513), (8, 30_000), (11, 12_345)):
        deg = _degrees("mixed", nnz, rng, short)
        deg = np.concatenate([deg, np.zeros(-len(deg) % 4, dtype=np.int64)])
        m, n = (short, len(deg)) if layout == "csc" else (len(deg), short)
        A = synth.random_matrix(m, n, layout, degrees=deg, seed=k, duplicates=True)
        plan, stored = make_plan(A, dtype, tile_items=256)
        for op, ln, ref, scale in ((pkg.SPMV_OP_AX, n, oracle.spmv, oracle.abs_spmv),
                                   (pkg.SPMV_OP_VTA, m, oracle.spvtm, oracle.abs_spvtm)):
            Z = torch.stack([dev_vec(synth.uniform_vector(ln, 10 + b), torch.float32) for b in range(k)])
            R = plan.batch(op, Z)
            plan.check()
            dots = (op == pkg.SPMV_OP_VTA) == (layout == "csc")
            for b in range(k):
                z = host_of(Z[b])
                assert_close(host_of(R[b]), ref(stored, z), scale(stored, z), TOL[dtype], f"{layout} {op} k={k} vector {b}")
                if dots:
                    assert torch.equal(R[b], plan.spvtm(Z[b]) if op == pkg.SPMV_OP_VTA else plan.spmv(Z[b]))


@pytest.mark.parametrize("layout", ["csc", "csr"])
@pytest.mark.parametrize("short,k", [(5_500, 8), (6_252, 8), (11_400, 4), (22_500, 2), (25_500, 2)])
def test_several_vectors_beside_few_warps(short, k, layout):
    """CTAs with tiles for all their warps, and accumulators or interleaved vectors that leave room for
    some of them only: the batch against the oracle, its dot products the single ones' bits."""
    rng = np.random.default_rng(short)
    deg = rng.integers(0, 80, 32_000)  # 1.26M nonzeros: 32 tiles a CTA
    m, n = (short, len(deg)) if layout == "csc" else (len(deg), short)
    A = synth.random_matrix(m, n, layout, degrees=deg, seed=k, duplicates=True)
    plan, stored = make_plan(A, torch.float32, tile_items=256)
    for op, ln, ref, scale in ((pkg.SPMV_OP_AX, n, oracle.spmv, oracle.abs_spmv),
                               (pkg.SPMV_OP_VTA, m, oracle.spvtm, oracle.abs_spvtm)):
        Z = torch.stack([dev_vec(synth.uniform_vector(ln, 10 + b), torch.float32) for b in range(k)])
        R = plan.batch(op, Z)
        plan.check()
        for b in range(k):
            z = host_of(Z[b])
            assert_close(host_of(R[b]), ref(stored, z), scale(stored, z), TOL[torch.float32], f"{layout} {op} vector {b}")
            if (op == pkg.SPMV_OP_VTA) == (layout == "csc"):
                assert torch.equal(R[b], plan.spvtm(Z[b]) if op == pkg.SPMV_OP_VTA else plan.spmv(Z[b]))


def test_row_blocks_in_turn():
    """Windows of the long vector too wide for one block a CTA: several blocks in turn, each restaging
    its window; the same bits as the streaming kernel's multi-vector pass over the same copy."""
    rng = np.random.default_rng(12)
    n = 5_000_000
    deg = np.zeros(n, dtype=np.int64)
    deg[rng.choice(n, 900_000, replace=False)] = 1
    deg[rng.choice(n, 20, replace=False)] = 64
    A = synth.random_matrix(64, n, "csc", degrees=deg, seed=3, duplicates=True)
    for dtype in (torch.float64, torch.float32):
        plan, stored = make_plan(A, dtype, flags=pkg.SPMV_PLAN_ROW_BLOCKS, tile_items=256)
        info = plan.info()
        if dtype == torch.float64:
            assert info["row_blocks"] > info["ctas"], info
        check_products(plan, stored, synth.uniform_vector(n, 1), synth.uniform_vector(64, 2), TOL[dtype], f"{dtype}")
        X = torch.stack([dev_vec(synth.uniform_vector(n, 7 + b), plan.vec_dtype) for b in range(2)])
        Y = plan.batch(pkg.SPMV_OP_AX, X)
        for b in range(2):
            assert torch.equal(Y[b], plan.spmv(X[b]))
        plan.close()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=str)
@pytest.mark.parametrize("m,n,blocks_in_turn", [(64, 9_000_000, True), (300, 400_000, False), (2_000, 60_000, False)])
def test_row_blocks_of_several_vectors(m, n, blocks_in_turn, dtype):
    """Batches over the row-sorted copy, windows on chip and read through L2, one block a CTA and several
    in turn: every vector the single product's bits."""
    rng = np.random.default_rng(m)
    deg = np.zeros(n, dtype=np.int64)
    deg[rng.choice(n, min(n, 1_500_000) * 9 // 10, replace=False)] = 1
    deg[rng.choice(n, min(n, 40_000), replace=False)] += int(max(2, 8 * 152 * m * 1.3 // 40_000))
    A = synth.random_matrix(m, n, "csc", degrees=deg, seed=3, duplicates=True)
    plan, stored = make_plan(A, dtype, flags=pkg.SPMV_PLAN_ROW_BLOCKS, tile_items=256)
    info = plan.info()
    assert info["row_blocks"] > 0 and (info["row_blocks"] > info["ctas"]) == blocks_in_turn, info
    X = torch.stack([dev_vec(synth.uniform_vector(n, 7 + b), torch.float32) for b in range(9)])
    single = [plan.spmv(X[b]) for b in range(9)]
    for k in (2, 3, 4, 7, 9):
        Y = plan.batch(pkg.SPMV_OP_AX, X[:k])
        plan.check()
        for b in range(k):
            assert torch.equal(Y[b], single[b]), f"k={k} vector {b}"
