"""The clustering's one-launch rounds at the edges of their tiles (224 clusters
and 16 neighbours on either side), where the last block takes over (1,024), and
with boxes whose union areas overflow: the tree holds every primitive once and
its boxes hold their primitives; where distances are finite it walks exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_12392_gb300 import rcp, scenes  # noqa: E402
import gpu_util as U  # noqa: E402

pytestmark = pytest.mark.gpu


def _walk(g, o, d, brute):
    m = len(o)
    ot = torch.from_numpy(np.concatenate([o, np.full((m, 1), 1e-4)], 1).astype(np.float32)).cuda()
    dt = torch.from_numpy(np.concatenate([d, np.full((m, 1), np.inf)], 1).astype(np.float32)).cuda()
    t = torch.empty(m, device="cuda")
    ids = torch.empty(m, dtype=torch.int32, device="cuda")
    rcp.rcp_debug_trace(g, m, ot, dt, 0, brute, t, ids)
    return t, ids


@pytest.mark.parametrize("n", [2, 15, 16, 17, 33, 65, 513, 1024, 1025, 1119, 1120, 1121, 1344, 9_633])
@pytest.mark.parametrize("spheres", [0, 3])
@pytest.mark.parametrize("scale", [1.0, 1e24])
def test_tree_over_tile_edges(n, spheres, scale):
    sc = scenes.random_soup(n, spheres, seed=n, tri_size=0.3)
    sc.tris *= np.float32(scale)  # 1e24: every union area is infinite
    sc.spheres *= np.float32(scale)
    g = U.gpu_scene(sc, rcp.RCP_COLLAPSE_AREA, 0)
    try:
        info = rcp.rcp_scene_get_info(g)
        assert info.n_records == n + spheres and info.max_leaf <= 3
        rcp.rcp_scene_validate(g)
        if scale != 1.0:
            return
        rng = np.random.default_rng(n)
        o = rng.uniform(-20, 20, (2000, 3)).astype(np.float32)
        d = sc.tris.reshape(-1, 3)[rng.integers(0, 3 * n, 2000)] - o
        d /= np.maximum(np.linalg.norm(d, axis=1, keepdims=True), 1e-6)
        walk, brute = _walk(g, o, d, 0), _walk(g, o, d, 1)
        assert torch.equal(walk[0], brute[0]) and torch.equal(walk[1], brute[1])
    finally:
        rcp.rcp_scene_destroy(g)


def test_near_ties_keep_their_tree():
    """A terrain's grid has many pairs whose union areas differ in the last bit:
    the order in which the area is rounded shows in the tree (46,969 nodes with
    the other order of its products)."""
    g = rcp.scene_from(scenes.terrain_scene(389))
    try:
        assert rcp.rcp_scene_get_info(g).n_nodes == 48_170
    finally:
        rcp.rcp_scene_destroy(g)
