"""Which multi-sample kernel a launch takes, served or not: the one with fewer
warps and nothing spilled up to 64 tiles per SM, the other above, whatever a
warp claims at once."""
import re

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_12392_gb300 import rcp, scenes  # noqa: E402
import gpu_util as U  # noqa: E402

pytestmark = pytest.mark.gpu

JIT = np.array([[0.2, 0.6], [0.7, 0.1]], np.float32)
MANY, FEW = 1, 2


def _variants(work):
    """The sample variants (fourth template argument) of the trace kernels that work() launches."""
    for _ in range(3):  # a process's first trace can come back empty
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            work()
            torch.cuda.synchronize()
        names = [e.name for e in prof.events()]
        if names:
            break
    else:
        pytest.skip("kernels cannot be traced here")
    return [int(m.group(1)) for m in (re.search(r"k_trace<\d+, \w+, \w+, (\d)", n) for n in names) if m]


def _line_rows():
    """Rows of 64-tile-wide images at the line."""
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.fixture(scope="module")
def scene():
    sc = scenes.tiny_scene()
    g = U.gpu_scene(sc)
    yield sc, g
    rcp.rcp_scene_destroy(g)


@pytest.mark.parametrize("chunk", [32, 64])
@pytest.mark.parametrize("rows,want", [(1, FEW), (0, FEW), (-1, MANY)])
def test_line_is_in_tiles(scene, chunk, rows, want):
    sc, g = scene
    rcp.rcp_set_tuning(g, rcp.rcp_tuning(block=128, chunk=chunk, fused_camera=1, stack_entries=0, hints=3,
                                         chain_passes=1))
    p = rcp.make_params(rcp.RCP_MAP_EYE, 0.05 * sc.diameter(), 6.0, jitter=JIT)
    W, H = 64 * 8, 4 * (_line_rows() if rows == 0 else _line_rows() + 1 if rows < 0 else rows)
    out = torch.empty((H, W, 4), device="cuda")
    cam = rcp.camera_from(sc.poses[0])
    assert _variants(lambda: rcp.rcp_render_device(g, cam, W, H, 1, p, None, out, None,
                                                   torch.cuda.current_stream())) == [want]


@pytest.mark.parametrize("rows,want", [(1, FEW), (0, FEW), (-1, MANY)])
def test_served_launches_follow_the_line(scene, rows, want):
    sc, g = scene
    p = rcp.make_params(rcp.RCP_MAP_EYE, 0.05 * sc.diameter(), 6.0, jitter=JIT)
    W, H = 64 * 8, 4 * (_line_rows() if rows == 0 else _line_rows() + 1 if rows < 0 else rows)
    cam = rcp.camera_from(sc.poses[0])
    out = np.empty((H, W, 3), np.float32)
    srv = rcp.rcp_server_create(1 << 30, 2)
    try:
        def serve():
            rcp.rcp_server_wait(srv, rcp.rcp_server_submit(srv, g, cam, W, H, 2, p, out), 60.0)

        assert _variants(serve) == [want] * 2
    finally:
        rcp.rcp_server_destroy(srv)
    assert np.array_equal(out, rcp.rcp_render(g, cam, W, H, 2, p))
