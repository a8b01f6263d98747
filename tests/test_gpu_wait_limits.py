"""Bounded waits of the sort and the build that run out: a status comes back, nothing is
followed that was not written, and the device stays usable."""
import pytest

torch = pytest.importorskip("torch")

from paper_2312_12392_gb300 import rcp, scenes  # noqa: E402
import gpu_util as U  # noqa: E402

pytestmark = pytest.mark.gpu


def _build_and_walk():
    sc = scenes.random_soup(9_633, 3, seed=5, tri_size=0.3)
    g = U.gpu_scene(sc)
    try:
        rcp.rcp_scene_validate(g)
        ot, dt = U.random_rays(2000, seed=3, extent=10.0, towards=(0, 0, 0))
        o, d = torch.from_numpy(ot).cuda(), torch.from_numpy(dt).cuda()
        res = []
        for brute in (0, 1):
            t, ids = torch.empty(2000, device="cuda"), torch.empty(2000, dtype=torch.int32, device="cuda")
            rcp.rcp_debug_trace(g, 2000, o, d, 0, brute, t, ids)
            res.append((t, ids))
        assert torch.equal(res[0][0], res[1][0]) and torch.equal(res[0][1], res[1][1])
    finally:
        rcp.rcp_scene_destroy(g)


@pytest.mark.parametrize("limit", [1, 1000, 100_000])
def test_clustering_wait(limit):
    with pytest.raises(rcp.RcpError) as e:
        rcp.rcp_debug_cluster_lookback_timeout(limit)
    assert e.value.status == rcp.RCP_ERR_TIMEOUT and "clustering" in str(e.value) and "ran out" in str(e.value)
    _build_and_walk()


@pytest.mark.parametrize("limit", [1, 1000, 100_000])
def test_barrier_wait(limit):
    with pytest.raises(rcp.RcpError) as e:
        rcp.rcp_debug_sort_barrier_timeout(limit)
    assert e.value.status == rcp.RCP_ERR_TIMEOUT and "ran out" in str(e.value)
    _build_and_walk()


@pytest.mark.parametrize("entry", [rcp.rcp_debug_cluster_lookback_timeout, rcp.rcp_debug_sort_barrier_timeout])
@pytest.mark.parametrize("limit", [0, (1 << 20) + 1])
def test_limits_are_checked(entry, limit):
    with pytest.raises(rcp.RcpError) as e:
        entry(limit)
    assert e.value.status == rcp.RCP_ERR_ARG
