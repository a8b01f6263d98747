"""Multi-sample renders that leave out tiles whose values repeat: image, hit
ids and ray counts equal those of one-pass renders chained by hand, which
trace every tile, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_12392_gb300 import rcp, scenes  # noqa: E402
import gpu_util as U  # noqa: E402

pytestmark = pytest.mark.gpu

JIT = np.array([[0.2, 0.6], [0.7, 0.1], [0.4, 0.9]], np.float32)


@pytest.fixture(scope="module", params=["tiny", "terrain"])
def scene(request):
    sc = scenes.tiny_scene() if request.param == "tiny" else scenes.terrain_scene(48, n_boxes=20)
    g = U.gpu_scene(sc)
    yield sc, g
    rcp.rcp_scene_destroy(g)


def _by_hand(g, cam, W, H, K, p, first, stream):
    """K one-pass renders; every pass's image, ids and ray counts."""
    img, out, rays = first, [], np.zeros(2, np.int64)
    for _ in range(K):
        nxt = torch.empty((H, W, 4), device="cuda")
        ids = torch.empty((H, W), dtype=torch.int32, device="cuda")
        rcp.rcp_render_device(g, cam, W, H, 1, p, img, nxt, ids, stream)
        torch.cuda.synchronize()
        rays = rays + np.array(rcp.rcp_last_ray_counts(g))
        out.append((nxt, ids, tuple(int(x) for x in rays)))
        img = nxt
    return out


@pytest.mark.parametrize("mapping,k_frac", [(rcp.RCP_MAP_EYE, 0.02), (rcp.RCP_MAP_EYE, 0.0), (rcp.RCP_MAP_TARGET, 0.02),
                                            (rcp.RCP_MAP_TARGET, 0.0), (rcp.RCP_MAP_DEPTH, 0.001),
                                            (rcp.RCP_MAP_NORMAL, 0.02)])
@pytest.mark.parametrize("W,H", [(67, 45), (8, 4), (1, 1), (129, 30)])
@pytest.mark.parametrize("spp", [1, 3])
def test_repeats_match_traced_passes(scene, mapping, k_frac, W, H, spp):
    sc, g = scene
    st = torch.cuda.current_stream()
    cam = rcp.camera_from(sc.poses[0])
    d = sc.diameter()
    p = rcp.make_params(mapping, k_frac * d, 0.1 * d, z0=0.1 * d, jitter=JIT[:spp])
    hand = _by_hand(g, cam, W, H, 9, p, None, st)
    for K in (1, 2, 3, 4, 5, 6, 9):
        for with_ids in (True, False, True):
            out = torch.full((H, W, 4), -1.0, device="cuda")
            ids = torch.full((H, W), -7, dtype=torch.int32, device="cuda") if with_ids else None
            rcp.rcp_render_device(g, cam, W, H, K, p, None, out, ids, st)
            torch.cuda.synchronize()
            assert torch.equal(out.view(torch.int32), hand[K - 1][0].view(torch.int32))
            assert rcp.rcp_last_ray_counts(g) == hand[K - 1][2]
            if with_ids:
                assert torch.equal(ids, hand[K - 1][1])
    # a given first image, rendered in place; and the host's RGB
    again = _by_hand(g, cam, W, H, 5, p, hand[1][0], st)
    out = hand[1][0].clone()
    rcp.rcp_render_device(g, cam, W, H, 5, p, out, out, None, st)
    torch.cuda.synchronize()
    assert torch.equal(out.view(torch.int32), again[4][0].view(torch.int32))
    assert np.array_equal(rcp.rcp_render(g, cam, W, H, 6, p), hand[5][0].cpu().numpy()[..., :3])


def test_views_of_a_batch_keep_their_own_repeats(scene):
    sc, g = scene
    st = torch.cuda.current_stream()
    d = sc.diameter()
    p = rcp.make_params(rcp.RCP_MAP_TARGET, 0.02 * d, 0.1 * d, jitter=JIT)
    cams = [rcp.camera_from(sc.poses[i % len(sc.poses)]) for i in (0, 7, 19)]
    sizes = [(67, 45), (9, 130), (64, 32)]
    outs = [torch.empty((h, w, 4), device="cuda") for w, h in sizes]
    ids = [torch.empty((h, w), dtype=torch.int32, device="cuda") for w, h in sizes]
    rcp.rcp_render_batch_device(g, cams, [w for w, _ in sizes], [h for _, h in sizes], 6, p, outs, st,
                                d_prims=[ids[0], None, ids[2]])
    torch.cuda.synchronize()
    for i, (w, h) in enumerate(sizes):
        hand = _by_hand(g, cams[i], w, h, 6, p, None, st)[5]
        assert torch.equal(outs[i].view(torch.int32), hand[0].view(torch.int32))
        assert i == 1 or torch.equal(ids[i], hand[1])
