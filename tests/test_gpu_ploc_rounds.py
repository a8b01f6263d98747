"""The clustering at the sizes where its rounds change form: one block up to
2,048 references, then tiles of 1,024 merged in one pass each. The tree holds
every primitive once and walks exactly, also for runs of equal boxes (there
to the distance: which of many equal triangles is named is not compared)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_12392_gb300 import rcp, scenes  # noqa: E402
import gpu_util as U  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 31, 1023, 1025, 2047, 2048, 2049, 3073, 40_001])
@pytest.mark.parametrize("kind", ["soup", "equal"])
@pytest.mark.parametrize("collapse,split", [(rcp.RCP_COLLAPSE_AREA, 0), (rcp.RCP_COLLAPSE_SAH, 8)])
def test_tree_is_whole_and_exact(n, kind, collapse, split):
    sc = scenes.random_soup(n, 0, seed=n, tri_size=0.3)
    if kind == "equal":  # every box the same
        sc.tris[:] = sc.tris[0]
    g = U.gpu_scene(sc, collapse, split)
    try:
        info = rcp.rcp_scene_get_info(g)
        assert info.n_records >= n and info.max_leaf <= 3
        rcp.rcp_scene_validate(g)
        if info.depth > 64:  # the surface-area collapse of equal boxes: deeper than a walk's stack, refused
            return
        rng = np.random.default_rng(n)
        m = 2000
        o = rng.uniform(-20, 20, (m, 3)).astype(np.float32)
        d = sc.tris.reshape(-1, 3)[rng.integers(0, 3 * n, m)] - o
        d /= np.maximum(np.linalg.norm(d, axis=1, keepdims=True), 1e-6)
        ot = torch.from_numpy(np.concatenate([o, np.full((m, 1), 1e-4)], 1).astype(np.float32)).cuda()
        dt = torch.from_numpy(np.concatenate([d, np.full((m, 1), np.inf)], 1).astype(np.float32)).cuda()
        got = []
        for brute in (0, 1):
            t = torch.empty(m, device="cuda")
            ids = torch.empty(m, dtype=torch.int32, device="cuda")
            rcp.rcp_debug_trace(g, m, ot, dt, 0, brute, t, ids)
            got.append((t, ids))
        assert torch.equal(got[0][0], got[1][0])
        if kind == "soup":  # a tie of equal triangles may lie outside the slack of a grazing hit's far limit
            assert torch.equal(got[0][1], got[1][1])
    finally:
        rcp.rcp_scene_destroy(g)
