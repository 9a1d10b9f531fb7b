"""The bytes that serving reserves for a host matrix before it plans it: never fewer than the plan then holds, and
no more than the lists of empty segments above that (host code over a fake CUDA runtime, CPU only)."""
import ctypes

import numpy as np
import pytest

from host_lib import BF16, F32, F64, HostLib
from paper_1812_00904_gb300 import _lib


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    host = HostLib(str(tmp_path_factory.mktemp("host")))
    host.lib.fake_plan_bytes_most.restype = ctypes.c_uint64
    host.lib.fake_plan_bytes_most.argtypes = [ctypes.c_int64] * 3 + [ctypes.c_int] * 2
    host.lib.spmv_plan_info.argtypes = [ctypes.c_void_p, ctypes.c_void_p]
    return host


@pytest.mark.parametrize("val", [F32, BF16, F64])
@pytest.mark.parametrize("m,n,nnz", [(300, 5_000, 40_000), (2_000, 150_000, 3_000_000), (45_000, 1_000, 100_000),
                                     (60_000, 40_000, 500_000), (4_000, 2_000_000, 60_000), (8_000, 500, 0),
                                     (1_500, 1_000_000, 20_000_000)])
@pytest.mark.parametrize("empty", [False, True])
def test_reserved_bytes(host, val, m, n, nnz, empty):
    host.reset()
    if empty:
        ptr = np.minimum(np.arange(n + 1, dtype=np.int64) * 2 * nnz // n, nnz).astype(np.int32)  # (the later half)
    else:
        ptr = (np.arange(n + 1, dtype=np.int64) * nnz // n).astype(np.int32)
    plan = host.plan(m, n, nnz, val, ptr=ptr)
    info = _lib.spmv_plan_info_t()
    assert host.lib.spmv_plan_info(plan, ctypes.byref(info)) == 0
    held = info.workspace_bytes + nnz * (4 + {F32: 4, BF16: 2, F64: 8}[val]) + 4 * (n + 1)
    host.close(plan)
    most = host.lib.fake_plan_bytes_most(m, n, nnz, val, F64 if val == F64 else F32)
    assert held <= most <= held + 8 * n + n // 64 + 64
    if np.any(np.diff(ptr) == 0):
        assert most == held or nnz == 0
