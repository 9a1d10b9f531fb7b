"""Which kernel a call on a validated plan goes to, and with how many warps, along the lines of the dispatch rules
(host code over a fake CUDA runtime, CPU only)."""
import pytest

from host_lib import BF16, F16, F32, F64, HostLib

SLOT = {F32: 2112, BF16: 1600, F16: 1600, F64: 3136}
MOST = {F32: 32, BF16: 32, F16: 32, F64: 16}
ROOM = 232448 - 1024 - 512


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    host = HostLib(str(tmp_path_factory.mktemp("host")))
    yield host


def m_for(val, warps, vectors=1):
    """The longest short vector (a multiple of 32 elements) beside which that many warps' slots fit."""
    return (ROOM - warps * SLOT[val]) // (8 if val == F64 else 4) // vectors // 32 * 32


@pytest.mark.parametrize("nnz", [5_000, 38_000, 400_000, 3_000_000, 30_000_000])
@pytest.mark.parametrize("val,warps", [(v, w) for v in (F32, BF16, F16, F64) for w in (1, 4, 7, 8, 12, 16, 20, 31, 32)
                                       if w <= MOST[v]])
def test_a_pass_has_the_warps_its_vectors_need(host, val, nnz, warps):
    most = MOST[val]
    host.reset()
    m = m_for(val, warps)
    plan = host.plan(m, 1_000, nnz, val)
    for call, name in (("spmv", "pass scatter"), ("spvtm", "pass segdot")):
        (kernel, w, ctas), *_ = host.launches(plan, call)
        if kernel == name:
            assert w == min(warps, most) >= 8  # (short vectors this long ask for all of them)
        else:
            assert kernel == name.replace("pass", "stream")
            assert warps < 8 or call == "spmv" and warps < most and nnz < max(0.55, 8.0 / warps) * ctas * m * 1.001
    host.close(plan)


@pytest.mark.parametrize("nnz,least", [(5_000, 8), (311_296, 8), (311_297, 12), (3_000_000, 12), (30_000_000, 20)])
@pytest.mark.parametrize("val,warps", [(v, w) for v in (F32, BF16, F64) for w in (1, 7, 8, 11, 12, 16, 19, 20, 32)
                                       if w <= MOST[v]])
def test_the_pair_is_one_pass_with_enough_warps(host, val, nnz, least, warps):
    least = min(least, MOST[val])
    host.reset()
    plan = host.plan(m_for(val, warps, vectors=2), 1_000, nnz, val)
    kernels = [k for k, _, _ in host.launches(plan, "spmv_pair")]
    assert ("pass pair" in kernels) == (warps >= least)
    host.close(plan)


@pytest.mark.parametrize("val,m", [(F32, 300), (F32, 40_000), (F64, 4_000)])
def test_short_vectors_with_room_for_all_warps_stay_on_chip(host, val, m):
    for nnz in (256, 5_000, 1_000_000):
        host.reset()
        plan = host.plan(m, 500, nnz, val)
        assert host.launches(plan, "spmv")[0][0] == "pass scatter"
        assert host.launches(plan, "spvtm")[0][0] == "pass segdot"
        assert host.launches(plan, "spmv_pair")[0][0] == ("pass pair" if m < 20_000 else "pass segdot")
        host.close(plan)


@pytest.mark.parametrize("m,nnz,launches", [(300, 4_877, 1), (4_000, 60_000, 2), (15_000, 5_000, 1), (12_000, 100_000, 4),
                                            (300, 233_472, 1), (300, 233_473, 0), (300, 8_000_000, 0)])
def test_f64_batches_of_small_matrices_take_a_pass_for_each_vector(host, m, nnz, launches):
    host.reset()
    plan = host.plan(m, 1_000, nnz, F64)
    kernels = [k for k, _, _ in host.launches(plan, "batch", 0, 8, 1_000, m)]
    assert kernels.count("pass scatter") == launches
    assert ("stream scatter" in kernels) == (launches == 0)
    host.close(plan)
