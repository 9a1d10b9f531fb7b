"""The shared memory that the blocks of the combine and fix-up kernel ask for: within the device's limit, all blocks
resident at once, none more to an SM than its share (host code, CPU only)."""
import ctypes
import re

import pytest

from host_lib import CSRC, HostLib


@pytest.fixture(scope="module")
def request_of(tmp_path_factory):
    lib = HostLib(str(tmp_path_factory.mktemp("host"))).lib
    lib.fake_finish_request.argtypes = [ctypes.c_int64, ctypes.c_int, ctypes.c_int]
    return lib.fake_finish_request


@pytest.mark.parametrize("sms,most", [(152, 232448), (148, 232448), (132, 232448), (64, 101376), (20, 49152)])
@pytest.mark.parametrize("blocks", [1, 19, 20, 21, 152, 153, 304, 626, 1063, 1064, 1065, 5000])
def test_request(request_of, sms, most, blocks):
    request, per_sm = request_of(blocks, sms, most), -(-blocks // sms)
    assert 0 <= request <= most - 2048  # (static memory of a block)
    used = request + 2048 + 1024        # (and what the system reserves for one)
    if request:
        assert per_sm * used <= most + 1024 < (per_sm + 1) * used or per_sm >= 6
    else:
        assert per_sm >= 8 or most // per_sm < 6144


def test_the_kernel_asks_for_it_with_its_own_device():
    text = open(f"{CSRC}/small_kernels.cu").read()
    assert "finish_request(blocks * kb, sms, most)" in text
    assert not re.search(r"\b(SMS|ALL)\b", text)
