"""A host matrix is admitted only where it fits the budget together with its plan."""
import numpy as np
import pytest
import torch

import synth
import paper_1812_00904_gb300 as pkg

pytestmark = pytest.mark.gpu


def admit(budget, host, m, n):
    """Resident bytes after a product of the matrix, or the status it fails with."""
    ptr, idx, vals = host
    srv = pkg.serve_create(budget, k_max=4, n_streams=1)
    try:
        mid = pkg.serve_register_host(srv, m, n, len(idx), pkg.SPMV_CSC_WIDE, ptr, idx, vals, pkg.SPMV_F32, pkg.SPMV_F32)
        x, y = torch.ones(n, device="cuda"), torch.empty(m, device="cuda")
        torch.cuda.synchronize()
        try:
            pkg.serve_wait(srv, pkg.serve_submit(srv, mid, pkg.SPMV_OP_AX, 1, x, y), 60_000)
        except pkg.SpmvError as e:
            return None, e.status
        assert abs(float(y.double().sum()) - float(vals.astype(np.float64).sum())) <= 1e-3 * len(idx)
        return pkg.serve_stats(srv)["resident_bytes"], 0
    finally:
        pkg.serve_destroy(srv)


# (the reservation counted 8 bytes a nonzero and no step records: the plan holds 0.45 bytes a nonzero beside
# that; and no lists of empty segments, 8 bytes each)
@pytest.mark.parametrize("m,n,nnz,every", [(200, 40_000, 20_000_000, 1), (2_000, 3_000_000, 600_000, 9)])
def test_no_admission_beyond_the_budget(m, n, nnz, every):
    rng = np.random.default_rng(m)
    cols = np.sort(rng.integers(0, n // every, nnz)) * every
    ptr = np.searchsorted(cols, np.arange(n + 1)).astype(np.int32)
    host = (ptr, rng.integers(0, m, nnz).astype(np.int32), rng.uniform(-1, 1, nnz).astype(np.float32))
    held, status = admit(1 << 34, host, m, n)
    assert status == 0
    assert admit(held - 1, host, m, n) == (None, 7)
    assert admit(held + 8 * n + (1 << 20), host, m, n) == (held, 0)
