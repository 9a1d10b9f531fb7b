"""The values' gradient with its minor vector on chip and, too long for it, in global memory: one product a nonzero,
rounded once to the accumulation type and once to the values' type, so exact."""
import numpy as np
import pytest
import torch

import paper_1812_00904_gb300 as pkg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", ["csc", "csr"])
@pytest.mark.parametrize("dtype,minor", [
    (torch.float32, 300), (torch.float32, 53_400), (torch.float32, 57_500), (torch.float32, 200_001), (torch.bfloat16, 60_000),
    (torch.float16, 70_001), (torch.float64, 25_600), (torch.float64, 30_000), (torch.float64, 200_001),
], ids=str)
@pytest.mark.parametrize("nnz", [1, 255, 256, 130_001, 3_000_007])
def test_gradient_is_exact(dtype, minor, nnz, layout):
    major = max(3, nnz // 2)  # (short and empty segments)
    gen = torch.Generator(device="cuda").manual_seed(nnz + minor)
    ptr = torch.randint(0, nnz + 1, (major + 1,), generator=gen, device="cuda").sort().values.to(torch.int32)
    ptr[0], ptr[-1] = 0, nnz
    idx = torch.randint(0, minor, (nnz,), generator=gen, device="cuda", dtype=torch.int32)
    vals = torch.rand(nnz, generator=gen, device="cuda", dtype=torch.float64).to(dtype)
    m, n = (minor, major) if layout == "csc" else (major, minor)
    vec = torch.float64 if dtype == torch.float64 else torch.float32
    plan = pkg.Plan(m, n, ptr, idx, vals, layout=layout)
    r = torch.randn(m, generator=gen, device="cuda", dtype=vec)
    x = torch.randn(n, generator=gen, device="cuda", dtype=vec)
    out = torch.full((nnz + 16,), 7.0, device="cuda", dtype=dtype)
    plan.dvalues(r, x, out=out[:nnz])
    plan.check()
    seg = torch.repeat_interleave(torch.arange(major, device="cuda"), (ptr[1:] - ptr[:-1]).long())
    want = (r[idx.long()] * x[seg] if layout == "csc" else r[seg] * x[idx.long()]).to(dtype)
    assert torch.equal(out[:nnz], want)
    assert bool((out[nnz:] == 7.0).all())  # (nothing behind the gradient is written)
    plan.close()
