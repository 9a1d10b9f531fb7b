"""Short vectors of a few elements (an accumulator element for every lane up to 32 of them, FP64 pairs up to 64), against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_1812_00904_gb300 as pkg
from gpu_util import TOL, assert_close, check_products, dev_vec, host_of, make_plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", ["csc", "csr"])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float16, torch.float64], ids=str)
@pytest.mark.parametrize("minor", [1, 2, 3, 16, 31, 32, 33, 64, 65])
@pytest.mark.parametrize("nnz", [1, 255, 5_003, 600_001])
def test_products(minor, nnz, dtype, layout):
    major = max(4, nnz // 20 // 4 * 4)
    rng = np.random.default_rng(nnz + minor)
    ptr = np.sort(rng.integers(0, nnz + 1, major + 1)).astype(np.int32)
    ptr[0], ptr[-1] = 0, nnz
    m, n = (minor, major) if layout == "csc" else (major, minor)
    A = synth.SparseMatrix(layout, m, n, ptr, rng.integers(0, minor, nnz).astype(np.int32), rng.uniform(-1, 1, nnz))
    plan, stored = make_plan(A, dtype)
    x, v = synth.uniform_vector(n, 1), synth.uniform_vector(m, 2)
    check_products(plan, stored, x, v, TOL[dtype], "products")
    xd, vd = dev_vec(x, plan.vec_dtype), dev_vec(v, plan.vec_dtype)
    y, u = torch.empty(m, dtype=plan.vec_dtype, device="cuda"), torch.empty(n, dtype=plan.vec_dtype, device="cuda")
    pkg.spmv_pair(plan.handle, xd, y, vd, u)
    plan.check()
    xs, vs = host_of(xd), host_of(vd)
    assert_close(host_of(y), oracle.spmv(stored, xs), oracle.abs_spmv(stored, xs), TOL[dtype], "pair y")
    assert_close(host_of(u), oracle.spvtm(stored, vs), oracle.abs_spvtm(stored, vs), TOL[dtype], "pair u")
    if minor % 4 == 0:
        op = pkg.SPMV_OP_AX if layout == "csc" else pkg.SPMV_OP_VTA
        product, scale = (oracle.spmv, oracle.abs_spmv) if layout == "csc" else (oracle.spvtm, oracle.abs_spvtm)
        X = torch.stack([dev_vec(synth.uniform_vector(major, 5 + b), plan.vec_dtype) for b in range(5)])
        Y = host_of(plan.batch(op, X))
        plan.check()
        for b in range(5):
            xb = host_of(X[b])
            assert_close(Y[b], product(stored, xb), scale(stored, xb), TOL[dtype], f"vector {b}")
    plan.close()
