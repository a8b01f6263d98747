"""Renders of one shape on several streams and threads, which share the scene's
buffers for that shape: every frame equals the one rendered alone, bit for bit."""
import threading
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_12392_gb300 import rcp, scenes  # noqa: E402
import gpu_util as U  # noqa: E402

pytestmark = pytest.mark.gpu

JIT = np.array([[0.2, 0.6], [0.7, 0.1]], np.float32)
W, H, N = 1280, 720, 8

# mapping, K, samples, chained passes, views: one launch; two; one per pass (its
# first run, then its graph); the same with repeats; many descriptors
KINDS = {"chain": (rcp.RCP_MAP_EYE, 6, None, 1, 1), "image": (rcp.RCP_MAP_IMAGE, 4, None, 1, 1),
         "passes": (rcp.RCP_MAP_TARGET, 3, None, 0, 1), "samples": (rcp.RCP_MAP_EYE, 4, JIT, 1, 1),
         "batch": (rcp.RCP_MAP_NORMAL, 3, None, 1, 6)}


@pytest.fixture(scope="module")
def scene():
    sc = scenes.terrain_scene(48, n_boxes=20)
    g = U.gpu_scene(sc)
    yield sc, g
    rcp.rcp_scene_destroy(g)


class Job:
    def __init__(self, sc, g, kind):
        mapping, self.K, jit, chain, self.views = KINDS[kind]
        self.g, self.sc = g, sc
        d = sc.diameter()
        self.p = rcp.make_params(mapping, 8.0 if mapping == rcp.RCP_MAP_IMAGE else 0.02 * d, 0.1 * d, jitter=jit)
        rcp.rcp_set_tuning(g, rcp.rcp_tuning(block=128, chunk=32, fused_camera=1, stack_entries=0, hints=3,
                                             chain_passes=chain))

    def cams(self, i):
        return [rcp.camera_from(self.sc.poses[(5 * i + v) % len(self.sc.poses)]) for v in range(self.views)]

    def outs(self):
        return [torch.full((H, W, 4), -1.0, device="cuda") for _ in range(self.views)]

    def render(self, i, outs, stream):
        if self.views == 1:
            rcp.rcp_render_device(self.g, self.cams(i)[0], W, H, self.K, self.p, None, outs[0], None, stream)
        else:
            rcp.rcp_render_batch_device(self.g, self.cams(i), [W] * self.views, [H] * self.views, self.K, self.p, outs,
                                        stream)

    def alone(self):
        res = []
        for i in range(N):
            outs = self.outs()
            self.render(i, outs, torch.cuda.current_stream())
            torch.cuda.synchronize()
            res.append(outs)
        return res


def _same(a, b):
    return all(torch.equal(x.view(torch.int32), y.view(torch.int32)) for x, y in zip(a, b))


@pytest.mark.parametrize("kind", KINDS)
def test_streams_take_turns(scene, kind):
    job = Job(*scene, kind)
    got = [job.outs() for _ in range(N)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for i in range(N):
        job.render(i, got[i], streams[i % 2])
    torch.cuda.synchronize()
    ref = job.alone()
    assert [_same(a, b) for a, b in zip(got, ref)] == [True] * N


def test_host_render_behind_a_device_render(scene):
    job = Job(*scene, "chain")
    ref = job.alone()
    out = job.outs()
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    for i in range(0, N, 2):  # the second runs on the library's own stream
        job.render(i, out, st)
        host = rcp.rcp_render(job.g, job.cams(i + 1)[0], W, H, job.K, job.p)
        st.synchronize()
        assert _same(out, ref[i])
        assert np.array_equal(host, ref[i + 1][0].cpu().numpy()[..., :3])


@pytest.mark.parametrize("kind", ["chain", "passes"])
def test_threads_share_a_shape(scene, kind):
    job = Job(*scene, kind)
    got = [job.outs() for _ in range(N)]
    torch.cuda.synchronize()
    failed = []

    def work(t):
        try:
            st = torch.cuda.Stream()
            for i in range(t, N, 2):
                job.render(i, got[i], st)
        except Exception as e:  # noqa: BLE001
            failed.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed
    ref = job.alone()
    assert [_same(a, b) for a, b in zip(got, ref)] == [True] * N


@pytest.mark.parametrize("kind", ["chain", "samples"])
def test_first_render_of_a_shape_does_not_wait_for_the_legacy_stream(scene, kind):
    """The buffers made for a shape are cleared on the frame's own stream: a clear
    behind the legacy stream's work would land in or after the frame."""
    job = Job(*scene, kind)
    w, h = (611, 333) if kind == "chain" else (613, 335)  # shapes that nothing else here renders
    st = torch.cuda.Stream()
    img = torch.rand((h, w, 4), generator=torch.Generator().manual_seed(3)).cuda()
    first = img.clone()
    torch.cuda.synchronize()
    torch.cuda._sleep(100_000_000)  # about 50 ms of the legacy stream
    rcp.rcp_render_device(job.g, job.cams(0)[0], w, h, job.K, job.p, img, img, None, st)
    st.synchronize()
    rays = rcp.rcp_last_ray_counts(job.g)  # read behind the legacy stream's work
    torch.cuda.synchronize()
    assert rays[0] == w * h * job.K * max(job.p.spp, 1)
    out = torch.empty_like(first)
    rcp.rcp_render_device(job.g, job.cams(0)[0], w, h, job.K, job.p, first, out, None, st)
    torch.cuda.synchronize()
    assert rcp.rcp_last_ray_counts(job.g) == rays
    assert torch.equal(img.view(torch.int32), out.view(torch.int32))


def test_a_new_servers_counts_do_not_wait_for_the_legacy_stream(scene):
    sc, g = scene
    d = sc.diameter()
    p = rcp.make_params(rcp.RCP_MAP_EYE, 0.02 * d, 0.1 * d)
    torch.cuda.synchronize()
    torch.cuda._sleep(200_000_000)
    srv = rcp.rcp_server_create(1 << 30, 2)
    try:
        out = np.zeros((90, 160, 3), np.float32)
        t = rcp.rcp_server_submit(srv, g, rcp.camera_from(sc.poses[0]), 160, 90, 4, p, out)
        rcp.rcp_server_wait(srv, t, 60.0)
        time.sleep(0.1)  # the step's end, where its rays are added up
        s = rcp.rcp_server_stats_get(srv)
        assert s.mrays_per_s / s.frames_per_s * 1e6 >= 0.999 * 160 * 90 * 4
    finally:
        rcp.rcp_server_destroy(srv)


@pytest.mark.parametrize("chain", [0, 1])
def test_shapes_on_two_streams_share_the_stack_region(scene, chain):
    """A shared stack of one entry spills to a region of the scene that launches of
    every shape use."""
    job = Job(*scene, "chain")
    rcp.rcp_set_tuning(job.g, rcp.rcp_tuning(block=128, chunk=32, fused_camera=1, stack_entries=1, hints=3,
                                             chain_passes=chain))
    sizes = [(W, H), (W - 8, H)]
    outs = [torch.empty((h, w, 4), device="cuda") for w, h in sizes for _ in range(4)]
    refs = [torch.empty_like(o) for o in outs]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for alone, res in ((False, outs), (True, refs)):
        for i in range(4):
            for v, (w, h) in enumerate(sizes):
                rcp.rcp_render_device(job.g, job.cams(i + v)[0], w, h, job.K, job.p, None, res[4 * v + i], None,
                                      streams[v])
                if alone:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
    assert [_same([a], [b]) for a, b in zip(outs, refs)] == [True] * 8
