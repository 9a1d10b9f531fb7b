"""Plan memory from the pool and, for large blocks, beside it: what a closed plan held can be had again."""
import numpy as np
import pytest
import torch

import paper_1812_00904_gb300 as pkg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nnz", [1_000_000, 40_000_000])  # the bank-ordered copy: 8 and 320 MB
def test_closed_plans_give_their_memory_back(nnz):
    n, m = nnz // 20, 1_000
    ptr = torch.arange(0, nnz + 1, 20, dtype=torch.int32, device="cuda")
    idx = (torch.arange(nnz, dtype=torch.int32, device="cuda") * 7) % m
    vals = torch.ones(nnz, device="cuda")
    v = torch.ones(m, device="cuda")
    free = None
    for turn in range(5):
        plan = pkg.Plan(m, n, ptr, idx, vals, layout="csc", flags=pkg.SPMV_PLAN_BANK_ORDER)
        u = plan.spvtm(v)
        plan.check()
        plan.close()
        assert np.all(u.cpu().numpy() == 20.0)
        torch.cuda.synchronize()
        left = torch.cuda.mem_get_info()[0]
        free = left if free is None else free
        # (a pool keeps at most 512 MB; a plan that leaked its copy would take 1.3 GB by the fifth turn)
        assert left >= free - (512 << 20), f"turn {turn}: {(free - left) >> 20} MB less than after the first plan"
