"""The accumulating product with its short vector in global memory although the dot products keep theirs on chip
(long short vectors, few nonzeros), against the oracle over the forms that a plan accepts."""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_1812_00904_gb300 as pkg
from gpu_util import TOL, assert_close, check_products, dev_vec, host_of, make_plan

pytestmark = pytest.mark.gpu


# (FP32 45,000 and 52,000 elements leave the pass 24 and 11 of 32 warps, FP64 24,000 12 of 16; the line lies at
# 3.9M, 5.7M and 2.3M nonzeros)
@pytest.mark.parametrize("layout", ["csc", "csr"])
@pytest.mark.parametrize("dtype,minor,nnz", [
    (torch.float32, 45_000, 1), (torch.float32, 45_001, 100_003), (torch.float32, 52_000, 3_000_000),
    (torch.float32, 45_000, 5_000_000), (torch.bfloat16, 52_001, 700_001), (torch.float16, 45_000, 300_000),
    (torch.float64, 24_000, 255), (torch.float64, 24_002, 400_001), (torch.float64, 24_000, 3_000_000),
], ids=str)
@pytest.mark.parametrize("flags", [0, pkg.SPMV_PLAN_BANK_ORDER], ids=["stored", "bank"])
def test_products(dtype, minor, nnz, layout, flags):
    major = max(3, nnz // 30)
    rng = np.random.default_rng(nnz)
    ptr = np.sort(rng.integers(0, nnz + 1, major + 1)).astype(np.int32)  # (some segments empty)
    ptr[0], ptr[-1] = 0, nnz
    m, n = (minor, major) if layout == "csc" else (major, minor)
    A = synth.SparseMatrix(layout, m, n, ptr, rng.integers(0, minor, nnz).astype(np.int32), rng.uniform(-1, 1, nnz))
    plan, stored = make_plan(A, dtype, flags=flags)
    x, v = synth.uniform_vector(n, 1), synth.uniform_vector(m, 2)
    check_products(plan, stored, x, v, TOL[dtype], "products")
    xd, vd = dev_vec(x, plan.vec_dtype), dev_vec(v, plan.vec_dtype)
    y, u = torch.empty(m, dtype=plan.vec_dtype, device="cuda"), torch.empty(n, dtype=plan.vec_dtype, device="cuda")
    pkg.spmv_pair(plan.handle, xd, y, vd, u)
    plan.check()
    xs, vs = host_of(xd), host_of(vd)
    assert_close(host_of(y), oracle.spmv(stored, xs), oracle.abs_spmv(stored, xs), TOL[dtype], "pair y")
    assert_close(host_of(u), oracle.spvtm(stored, vs), oracle.abs_spvtm(stored, vs), TOL[dtype], "pair u")
    if m % 4 == 0 and n % 4 == 0:
        op = pkg.SPMV_OP_AX if layout == "csc" else pkg.SPMV_OP_VTA
        length = n if layout == "csc" else m
        X = torch.stack([dev_vec(synth.uniform_vector(length, 5 + b), plan.vec_dtype) for b in range(3)])
        Y = host_of(plan.batch(op, X))
        plan.check()
        product, scale = (oracle.spmv, oracle.abs_spmv) if layout == "csc" else (oracle.spvtm, oracle.abs_spvtm)
        for b in range(3):
            xb = host_of(X[b])
            assert_close(Y[b], product(stored, xb), scale(stored, xb), TOL[dtype], f"batch {b}")
    plan.close()
