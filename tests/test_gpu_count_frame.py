"""rcp_count_frame: the counters of a frame as its launches run it. The image is
the rendered one; passes left out because their values repeat are not counted."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_12392_gb300 import rcp, scenes  # noqa: E402
import gpu_util as U  # noqa: E402

pytestmark = pytest.mark.gpu

JIT = np.array([[0.2, 0.6], [0.7, 0.1]], np.float32)


@pytest.fixture(scope="module")
def scene():
    sc = scenes.terrain_scene(48, n_boxes=20)
    g = U.gpu_scene(sc)
    yield sc, g
    rcp.rcp_scene_destroy(g)


def _tuning(g, chain, fused=1, stack=0):
    rcp.rcp_set_tuning(g, rcp.rcp_tuning(block=128, chunk=32, fused_camera=fused, stack_entries=stack, hints=3,
                                         chain_passes=chain))


@pytest.mark.parametrize("mapping", [rcp.RCP_MAP_EYE, rcp.RCP_MAP_NORMAL, rcp.RCP_MAP_IMAGE])
@pytest.mark.parametrize("K", [1, 2, 5])
@pytest.mark.parametrize("chain,fused,stack", [(1, 1, 0), (0, 1, 0), (0, 0, 0), (1, 1, 1)])
@pytest.mark.parametrize("samples", [0, 2])
def test_same_frame_and_its_rays(scene, mapping, K, chain, fused, stack, samples):
    if mapping == rcp.RCP_MAP_IMAGE and samples:
        return
    sc, g = scene
    _tuning(g, chain, fused, stack)
    d = sc.diameter()
    W, H = 203, 77
    cam = rcp.camera_from(sc.poses[3])
    p = rcp.make_params(mapping, 8.0 if mapping == rcp.RCP_MAP_IMAGE else 0.02 * d, 0.1 * d,
                        jitter=JIT[:samples] if samples else None)
    ref, out = torch.empty((H, W, 4), device="cuda"), torch.empty((H, W, 4), device="cuda")
    rcp.rcp_render_device(g, cam, W, H, K, p, None, ref, None, torch.cuda.current_stream())
    torch.cuda.synchronize()
    primary, shadow = rcp.rcp_last_ray_counts(g)
    c = rcp.rcp_count_frame(g, cam, W, H, K, p, None, out)
    assert torch.equal(out.view(torch.int32), ref.view(torch.int32))
    assert c.rays == c.primary_rays + c.shadow_rays and 0 < c.primary_rays <= primary and c.shadow_rays <= shadow
    leaves_out = K > 2 if samples else chain and K > 1 and mapping != rcp.RCP_MAP_IMAGE
    if not leaves_out:
        assert (c.primary_rays, c.shadow_rays) == (primary, shadow)
    assert c.nodes >= c.rays and rcp.rcp_count_frame(g, cam, W, H, K, p).rays == c.rays


@pytest.mark.parametrize("samples", [0, 2])
def test_repeated_passes_are_not_counted(scene, samples):
    """With no displacement every pass from the second on repeats it."""
    sc, g = scene
    _tuning(g, 1)
    W, H, K = 64, 48, 6
    cam = rcp.camera_from(sc.poses[3])
    p = rcp.make_params(rcp.RCP_MAP_EYE, 0.0, 0.1 * sc.diameter(), jitter=JIT[:samples] if samples else None)
    one, two, all_ = (rcp.rcp_count_frame(g, cam, W, H, n, p) for n in (1, 2, K))
    assert all_.primary_rays == two.primary_rays == 2 * one.primary_rays == 2 * W * H * max(samples, 1)
    assert all_.shadow_rays == two.shadow_rays == 2 * one.shadow_rays


def test_arguments(scene):
    sc, g = scene
    cam = rcp.camera_from(sc.poses[3])
    buf = torch.zeros((8, 8, 4), device="cuda")
    for mapping, K, jit, d_out in ((rcp.RCP_MAP_EYE, 0, None, None), (rcp.RCP_MAP_EYE, 17, None, None),
                                   (rcp.RCP_MAP_IMAGE, 3, None, None), (rcp.RCP_MAP_EYE, 1, JIT, buf)):
        with pytest.raises(rcp.RcpError) as e:
            rcp.rcp_count_frame(g, cam, 8, 8, K, rcp.make_params(mapping, 0.1, 1.0, jitter=jit), buf, d_out)
        assert e.value.status == rcp.RCP_ERR_ARG
