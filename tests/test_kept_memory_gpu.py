"""Memory of closed plans on the device: nothing is lost over many plans, and what is kept goes back on request."""
import pytest
import torch

import paper_1812_00904_gb300 as pkg

pytestmark = pytest.mark.gpu


def made(kind):
    nnz, m, n = 1_000_000, 1_000, 50_000
    major = torch.arange(nnz, dtype=torch.int32, device="cuda") // 20
    if kind == "empty segments":
        major = major // 2 * 2  # (every other column empty: the lists of them)
    minor = (torch.arange(nnz, dtype=torch.int32, device="cuda") * 7) % m
    vals = torch.ones(nnz, device="cuda")
    ptr = torch.searchsorted(major, torch.arange(n + 1, dtype=torch.int32, device="cuda"), out_int32=True)
    v = torch.ones(m, device="cuda")

    def make():
        if kind == "unsorted triples":
            plan = pkg.Plan.from_coo(m, n, minor.flip(0), major.flip(0), vals, layout="csc", flags=pkg.SPMV_PLAN_COO_UNSORTED)
        else:
            flags = pkg.SPMV_PLAN_BANK_ORDER if kind == "bank order" else pkg.SPMV_PLAN_ROW_BLOCKS if kind == "row blocks" else 0
            plan = pkg.Plan(m, n, ptr, minor, vals, layout="csc", flags=flags)
        u = plan.spvtm(v)
        assert float(u.sum()) == nnz
        plan.close()

    return make


# (each plan holds 3 to 12 MB: 300 leaked ones would be more than the 512 MB kept at most)
@pytest.mark.parametrize("kind", ["stored order", "empty segments", "bank order", "row blocks", "unsorted triples"])
def test_many_plans_leave_the_memory_as_it_was(kind):
    make = made(kind)
    make()
    pkg.spmv_release_memory()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for _ in range(300):
        make()
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] >= free - (512 << 20)
    pkg.spmv_release_memory()
    assert torch.cuda.mem_get_info()[0] >= free - (32 << 20)  # (a leak of 100 kB a plan shows)
