"""The device sort of coordinate triples: one pass (which reads the triples and writes the sorted ones) and
several, at the edges of its 4096-key tiles, against a stable sort on the host.  Exact: nothing is computed."""
import numpy as np
import pytest
import torch

import paper_1812_00904_gb300 as pkg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float64], ids=str)
@pytest.mark.parametrize("n_minor,n_major,nnz", [
    (1, 1, 3),                 # no bits at all
    (1, 511, 4096), (512, 1, 4097), (20, 25, 1),  # one pass
    (3, 171, 4095),            # 513 keys: a second pass for one of them
    (700, 1500, 12_289),       # 21 bits
    (10_007, 500_009, 70_000),  # 33 bits
    (2**31 - 65, 3_000, 9_000),  # 43 bits, the largest minor dimension
    (1_000_003, 2_000_003, 40_000),  # 41 bits
])
def test_sorted_triples_equal_a_stable_host_sort(n_minor, n_major, nnz, dtype):
    rng = np.random.default_rng(nnz + n_minor)
    minor = rng.integers(0, n_minor, nnz).astype(np.int32)
    major = rng.integers(0, n_major, nnz).astype(np.int32)
    minor[-1], major[-1] = n_minor - 1, n_major - 1  # the largest key
    vals = torch.from_numpy(rng.standard_normal(nnz)).to(dtype)
    keys = major.astype(np.int64) * n_minor + minor
    perm = np.argsort(keys, kind="stable")
    dev = lambda a: torch.from_numpy(a).cuda()
    plan = pkg.Plan.from_coo(n_minor, n_major, dev(minor), dev(major), vals.cuda(), layout="csc",
                             flags=pkg.SPMV_PLAN_COO_UNSORTED)
    idx, got = plan.export()
    assert np.array_equal(idx.cpu().numpy(), minor[perm])
    assert torch.equal(got.cpu(), vals[torch.from_numpy(perm)])
    if n_major <= 1500:  # the pointer array, from the sorted major indices
        u = plan.spvtm(torch.ones(n_minor, dtype=torch.float64 if dtype == torch.float64 else torch.float32).cuda())
        plan.check()
        ref = np.bincount(major, weights=vals.double().numpy(), minlength=n_major)
        scale = np.bincount(major, weights=vals.double().abs().numpy(), minlength=n_major)
        tol = 1e-12 if dtype == torch.float64 else 1e-5
        assert np.all(np.abs(u.double().cpu().numpy() - ref) <= tol * scale)
