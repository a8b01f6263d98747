"""An image-space render's gathers in one launch equal one launch per pass, bit
for bit: ragged tiles, one-pixel images, displacements beyond the mirrored
edges, and batches of views."""
import pytest

torch = pytest.importorskip("torch")

from paper_2312_12392_gb300 import rcp, scenes  # noqa: E402
import gpu_util as U  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def scene():
    sc = scenes.terrain_scene(48, n_boxes=20)
    g = U.gpu_scene(sc)
    yield sc, g
    rcp.rcp_scene_destroy(g)


@pytest.mark.parametrize("sizes", [[(1, 1)], [(8, 4)], [(33, 5)], [(1, 300)], [(517, 203)], [(64, 64), (7, 9), (130, 61)]])
@pytest.mark.parametrize("kpx", [0.0, 6.0, 900.0, 3e9])
def test_one_launch_equals_one_per_pass(scene, sizes, kpx):
    sc, g = scene
    cam = rcp.camera_from(sc.poses[3])
    p = rcp.make_params(rcp.RCP_MAP_IMAGE, kpx, 0.1 * sc.diameter())
    for K in (1, 2, 3, 16):
        got = []
        for chain in (1, 0):
            t = rcp.rcp_get_tuning(g)
            t.chain_passes = chain
            rcp.rcp_set_tuning(g, t)
            outs = [torch.full((h, w, 4), -1.0, device="cuda") for w, h in sizes]
            rcp.rcp_render_batch_device(g, [cam] * len(sizes), [w for w, _ in sizes], [h for _, h in sizes], K, p, outs)
            torch.cuda.synchronize()
            assert len(rcp.rcp_last_pass_times(g)) == (K if not chain else min(K, 2))
            got.append(outs)
        for a, b in zip(*got):
            assert torch.equal(a.view(torch.int32), b.view(torch.int32))
