"""Segment counts up to the largest accepted (2^31 - 65): the index arithmetic of the kernels that list the empty
segments and zero their outputs (host code, CPU only; no GPU run at that size)."""
import ctypes
import re

import pytest

from host_lib import CSRC, HostLib

MOST = 2**31 - 65
STEP = 152 * 1024  # threads of a pass


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    lib = HostLib(str(tmp_path_factory.mktemp("host"))).lib
    lib.fake_ranked_segments.restype = lib.fake_strided.restype = ctypes.c_int64
    lib.fake_strided.argtypes = [ctypes.c_int64] * 3 + [ctypes.c_void_p] * 2
    return lib


@pytest.mark.parametrize("n", [1, 511, 512, 513, 2**31 - 600, 2**31 - 512, 2**31 - 511, MOST])
def test_every_segment_is_ranked_by_one_block(lib, n):
    blocks = lib.fake_rank_blocks(n)
    assert blocks == (n + 511) // 512
    low = ctypes.c_int64()
    for b in {0, blocks - 1}:
        assert lib.fake_ranked_segments(n, b, ctypes.byref(low)) == min(512, n - 512 * b)
        assert low.value == 512 * b


@pytest.mark.parametrize("n", [1, STEP, 2**31 - STEP, 2**31 - STEP + 1, MOST])
@pytest.mark.parametrize("thread", [0, 1, STEP - 1])
def test_strided_loops_stay_in_range(lib, n, thread):
    low, high = ctypes.c_int64(), ctypes.c_int64()
    seen = lib.fake_strided(thread, STEP, n, ctypes.byref(low), ctypes.byref(high))
    assert seen == len(range(thread, n, STEP))
    if seen:
        assert (low.value, high.value) == (thread, range(thread, n, STEP)[-1])


def test_the_kernels_loop_over_the_empty_segments_that_way():
    text = open(f"{CSRC}/pass_kernel.cuh").read()
    loops = re.findall(r"[^;{}]*p\.nempty[^;{}]*", text)
    assert len(loops) == 2 and all("strided((int64_t)blockIdx.x * blockDim.x" in s for s in loops)
    ranks = open(f"{CSRC}/plan.cu").read()
    assert ranks.count("const int64_t j0 = seg_rank_first(blockIdx.x, threadIdx.x);") == 2
