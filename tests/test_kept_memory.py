"""What the library keeps of closed plans' memory makes room for its own allocations, whether from the pool or beside
it, and goes back on request (host code over a fake CUDA runtime, CPU only)."""
import pytest

from host_lib import F32, HostLib


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    return HostLib(str(tmp_path_factory.mktemp("host")))


def keep(host):
    """Memory of closed plans in the pool and no other free device memory; the bytes kept."""
    host.reset()
    before = host.lib.fake_used()
    plans = [host.plan(40_000, 1_000, 3_000_000) for _ in range(2)]
    for p in plans:
        host.close(p)
    assert host.lib.fake_used() > before
    return host.lib.fake_used() - before


@pytest.mark.parametrize("call", [
    ("batch of dot products", "batch", 1, 2, 40_000, 1_000_000),  # the interleaved vectors, made on first use
    ("larger plan", None),
])
def test_kept_memory_makes_room(host, call):
    host.reset()
    plan = host.plan(40_000, 1_000_000, 1_500_000)
    kept = keep(host)
    host.lib.fake_room(0)
    if call[1]:
        assert host.launches(plan, *call[1:])[0][0] == "interleave"
    else:
        host.lib.fake_room(60 << 20)
        host.close(host.plan(40_000, 1_000_000, 6_000_000, F32))
    host.reset()
    host.close(plan)
    assert kept > 0


def test_kept_memory_goes_back_on_request(host):
    kept = keep(host)
    used = host.lib.fake_used()
    host.log()
    assert host.lib.spmv_release_memory() == 0
    assert "trim" in host.log()
    assert host.lib.fake_used() <= used - kept
