"""Multi-sample launches below and above the tile count where the kernel's
occupancy changes: views small on their own are rendered alone (few tiles) and
in a batch whose tiles together lie above the line; images and ids are equal."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_12392_gb300 import rcp, scenes  # noqa: E402
import gpu_util as U  # noqa: E402

pytestmark = pytest.mark.gpu

JIT = np.array([[0.2, 0.6], [0.7, 0.1], [0.4, 0.9], [0.9, 0.3]], np.float32)


@pytest.mark.parametrize("spp", [1, 2, 4])
@pytest.mark.parametrize("K", [1, 4])
@pytest.mark.parametrize("block", [64, 128, 256])
def test_few_tiles_equal_many(spp, K, block):
    sc = scenes.terrain_scene(48, n_boxes=20)
    g = U.gpu_scene(sc)
    try:
        rcp.rcp_set_tuning(g, rcp.rcp_tuning(block=block, chunk=32, fused_camera=1, stack_entries=0, hints=3, chain_passes=1))
        st = torch.cuda.current_stream()
        d = sc.diameter()
        p = rcp.make_params(rcp.RCP_MAP_TARGET, 0.02 * d, 0.1 * d, jitter=JIT[:spp])
        per_sm = torch.cuda.get_device_properties(0).multi_processor_count * 64
        sizes = [(131, 77), (8, 4), (1, 1), (8 * 64, 4 * (per_sm // 64 + 1))]  # the last alone lies above the line
        cams = [rcp.camera_from(sc.poses[i]) for i in (0, 7, 19, 3)]
        outs = [torch.empty((h, w, 4), device="cuda") for w, h in sizes]
        ids = [torch.empty((h, w), dtype=torch.int32, device="cuda") for w, h in sizes]
        rcp.rcp_render_batch_device(g, cams, [w for w, _ in sizes], [h for _, h in sizes], K, p, outs, st, d_prims=ids)
        for i, (w, h) in enumerate(sizes):
            img = torch.empty_like(outs[i])
            prim = torch.empty_like(ids[i])
            rcp.rcp_render_device(g, cams[i], w, h, K, p, None, img, prim, st)
            torch.cuda.synchronize()
            assert torch.equal(img.view(torch.int32), outs[i].view(torch.int32))
            assert torch.equal(prim, ids[i])
    finally:
        rcp.rcp_scene_destroy(g)
