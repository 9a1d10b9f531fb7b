"""Row-sorted blocks whose windows fit beside the staging of the pass that runs them, but not beside what the
streaming kernel's accumulating pass (which never runs on the copy) would stage."""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_1812_00904_gb300 as pkg
from gpu_util import TOL, assert_close, check_products, dev_vec, host_of, make_plan

pytestmark = pytest.mark.gpu


# (two nonzeros a column, 152 blocks: windows within half a tile, 256 columns, of n / 152)
@pytest.mark.parametrize("dtype,window,stages,lo,hi", [
    (torch.float64, 21_950, 0, 21_376, 22_576),
    (torch.float32, 39_400, 4, 38_000, 40_800),
], ids=["f64", "f32-4-stages"])
def test_windows_beside_the_pass(dtype, window, stages, lo, hi):
    m, n = 100, 152 * window
    rng = np.random.default_rng(window)
    idx = rng.integers(0, m, 2 * n).astype(np.int32)
    A = synth.SparseMatrix("csc", m, n, np.arange(0, 2 * n + 1, 2, dtype=np.int32), idx, rng.uniform(-1, 1, 2 * n))
    plan, stored = make_plan(A, dtype, flags=pkg.SPMV_PLAN_ROW_BLOCKS, stages=stages)
    info = plan.info()
    assert info["row_blocks"] == 152 and lo < info["row_block_window"] <= hi, info
    check_products(plan, stored, synth.uniform_vector(n, 1), synth.uniform_vector(m, 2), TOL[dtype], "windows")
    X = torch.stack([dev_vec(synth.uniform_vector(n, 3 + b), plan.vec_dtype) for b in range(3)])
    Y = plan.batch(pkg.SPMV_OP_AX, X)
    for b in range(3):
        x = host_of(X[b])
        assert_close(host_of(Y[b]), oracle.spmv(stored, x), oracle.abs_spmv(stored, x), TOL[dtype], f"batch {b}")
        assert torch.equal(Y[b], plan.spmv(X[b]))
    plan.check()
    plan.close()
