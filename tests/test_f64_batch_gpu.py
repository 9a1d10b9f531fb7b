"""FP64 batches in the accumulating direction, a pass for each vector in one launch (small matrices) and the
streaming kernel's pass over several beyond the line, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_1812_00904_gb300 as pkg
from gpu_util import TOL, assert_close, dev_vec, host_of, make_plan

pytestmark = pytest.mark.gpu


# (the line lies at 6 tiles of 256 for each of 152 CTAs: 233,472 nonzeros; 15,000 elements leave one vector a launch)
@pytest.mark.parametrize("layout", ["csc", "csr"])
@pytest.mark.parametrize("minor,nnz", [(2, 1), (2, 255), (300, 256), (300, 4_877), (1_000, 39_169), (4_000, 60_000),
                                       (8_000, 97_001), (15_000, 14_000), (300, 233_472), (300, 233_473)])
@pytest.mark.parametrize("k", [2, 3, 8, 9, 17])
def test_every_vector_of_a_batch(minor, nnz, layout, k):
    major = max(4, nnz // 20 // 4 * 4)
    rng = np.random.default_rng(nnz + k)
    ptr = np.sort(rng.integers(0, nnz + 1, major + 1)).astype(np.int32)
    ptr[0], ptr[-1] = 0, nnz
    m, n = (minor, major) if layout == "csc" else (major, minor)
    A = synth.SparseMatrix(layout, m, n, ptr, rng.integers(0, minor, nnz).astype(np.int32), rng.uniform(-1, 1, nnz))
    plan, stored = make_plan(A, torch.float64)
    op = pkg.SPMV_OP_AX if layout == "csc" else pkg.SPMV_OP_VTA
    product, scale = (oracle.spmv, oracle.abs_spmv) if layout == "csc" else (oracle.spvtm, oracle.abs_spvtm)
    X = torch.stack([dev_vec(synth.uniform_vector(major, 5 + b), torch.float64) for b in range(k)])
    Y = host_of(plan.batch(op, X))
    plan.check()
    for b in range(k):
        xb = host_of(X[b])
        assert_close(Y[b], product(stored, xb), scale(stored, xb), TOL[torch.float64], f"vector {b}")
    plan.close()
