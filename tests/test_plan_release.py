"""Destroying a plan waits for the device that owns its memory, whatever device is current, before the memory
goes back to the pool (host code over a fake CUDA runtime, CPU only)."""
import pytest

from host_lib import HostLib


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    return HostLib(str(tmp_path_factory.mktemp("host")))


@pytest.mark.parametrize("owner,current", [(0, 0), (1, 0), (0, 1), (3, 2)])
def test_destroy_waits_for_the_owning_device(host, owner, current):
    host.reset()
    host.device(owner)
    plan = host.plan(300, 5_000, 40_000)
    host.device(current)
    host.log()
    assert host.lib.spmv_plan_destroy(plan) == 0
    log = host.log()
    assert "pool free" in log
    assert f"sync device {owner}" in log[:log.index("pool free")]
    assert host.device() == current


def test_memory_stays_out_of_the_pool_when_the_wait_fails(host):
    """(A device that cannot be waited for, as while a stream of it is captured, may still run the plan's kernels.)"""
    host.reset()
    plan = host.plan(300, 5_000, 40_000)
    host.log()
    host.lib.fake_fail_sync(1)
    host.lib.spmv_plan_destroy(plan)
    assert "pool free" not in host.log()
    host.lib.fake_fail_sync(0)
    plan = host.plan(300, 5_000, 40_000)
    host.log()
    host.lib.spmv_plan_destroy(plan)
    log = host.log()
    assert log.count("pool free") == 4 and log[0] == "sync device 0"  # (both plans' two blocks)
