"""Chained renders whose pixels' values repeat (fixed points and cycles of two
passes): the image, hit ids and ray counts equal those of one launch per pass,
which traces every pass, bit for bit."""
import pytest

torch = pytest.importorskip("torch")

from paper_2312_12392_gb300 import rcp, scenes  # noqa: E402
import gpu_util as U  # noqa: E402

pytestmark = pytest.mark.gpu


def _render(g, cam, W, H, K, p, chain, first):
    t = rcp.rcp_get_tuning(g)
    t.chain_passes = chain
    rcp.rcp_set_tuning(g, t)
    out = torch.full((H, W, 4), -1.0, device="cuda")
    ids = torch.full((H, W), -7, dtype=torch.int32, device="cuda")
    rcp.rcp_render_device(g, cam, W, H, K, p, first, out, ids, torch.cuda.current_stream())
    torch.cuda.synchronize()
    return out.view(torch.int32), ids, rcp.rcp_last_ray_counts(g)


@pytest.mark.parametrize("mapping,k_frac", [(rcp.RCP_MAP_EYE, 0.02), (rcp.RCP_MAP_EYE, 0.0), (rcp.RCP_MAP_TARGET, 0.02),
                                            (rcp.RCP_MAP_DEPTH, 0.001), (rcp.RCP_MAP_NORMAL, 0.02)])
@pytest.mark.parametrize("scene", ["tiny", "terrain"])
def test_repeating_orbits_match_traced_passes(scene, mapping, k_frac):
    sc = scenes.tiny_scene() if scene == "tiny" else scenes.terrain_scene(48, n_boxes=20)
    g = U.gpu_scene(sc)
    try:
        cam = rcp.camera_from(sc.poses[0])
        d = sc.diameter()
        p = rcp.make_params(mapping, k_frac * d, 0.1 * d, z0=0.1 * d)
        W, H = 67, 45  # ragged tiles
        first = None
        for K in (1, 2, 3, 4, 7, 16):
            a, b = (_render(g, cam, W, H, K, p, chain, first) for chain in (1, 0))
            assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
            assert a[2] == b[2]
            if K == 7:  # continue from this image, whose orbits have partly closed
                last = b[0]
        if k_frac == 0.0:  # every pixel repeats from pass 2 on
            assert torch.equal(b[0], last)
        prev = last.view(torch.float32).clone()
        for K in (1, 2, 5):
            a, b = (_render(g, cam, W, H, K, p, chain, prev) for chain in (1, 0))
            assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and a[2] == b[2]
    finally:
        rcp.rcp_scene_destroy(g)
