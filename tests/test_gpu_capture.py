"""A render on a stream that is being captured is refused and leaves the caller's
capture, and the buffers of its shape, as they were."""
import pytest

torch = pytest.importorskip("torch")

from paper_2312_12392_gb300 import rcp, scenes  # noqa: E402
import gpu_util as U  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["global", "thread_local", "relaxed"])
@pytest.mark.parametrize("warm", [0, 1, 3])
@pytest.mark.parametrize("kind,K,chain", [("eye", 6, 1), ("eye", 1, 1), ("image", 3, 1), ("eye", 3, 0), ("samples", 3, 1)])
def test_refused_and_the_capture_goes_on(mode, warm, kind, K, chain):
    sc = scenes.tiny_scene()
    g = U.gpu_scene(sc)
    try:
        rcp.rcp_set_tuning(g, rcp.rcp_tuning(block=128, chunk=32, fused_camera=1, stack_entries=0, hints=3,
                                             chain_passes=chain))
        jit = [[0.2, 0.6], [0.7, 0.1]] if kind == "samples" else None
        image = kind == "image"
        p = rcp.make_params(rcp.RCP_MAP_IMAGE if image else rcp.RCP_MAP_EYE, 8.0 if image else 0.05 * sc.diameter(), 6.0,
                            jitter=jit)
        cam = rcp.camera_from(sc.poses[0])
        W, H = 75, 40
        out = torch.zeros((H, W, 4), device="cuda")
        mark = torch.zeros(8, device="cuda")
        st = torch.cuda.Stream()
        torch.cuda.synchronize()
        for _ in range(warm):
            rcp.rcp_render_device(g, cam, W, H, K, p, None, out, None, st)
        torch.cuda.synchronize()
        out.zero_()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st, capture_error_mode=mode):
            mark += 1
            with pytest.raises(rcp.RcpError) as e:
                rcp.rcp_render_device(g, cam, W, H, K, p, None, out, None, st)
            mark += 2
        assert e.value.status == rcp.RCP_ERR_CUDA and "captured" in str(e.value)
        graph.replay()
        torch.cuda.synchronize()
        assert (mark == 3).all() and not out.any()
        rcp.rcp_render_device(g, cam, W, H, K, p, None, out, None, st)
        ref = torch.empty_like(out)
        other = U.gpu_scene(sc)
        rcp.rcp_render_device(other, cam, W, H, K, p, None, ref, None, st)
        st.synchronize()
        rcp.rcp_scene_destroy(other)
        assert torch.equal(out.view(torch.int32), ref.view(torch.int32))
    finally:
        rcp.rcp_scene_destroy(g)
