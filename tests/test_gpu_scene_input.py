"""Scene arrays are checked and widened on the device: an infinity or NaN at any
coordinate is refused, at the ends of the arrays and at lengths that leave a
remainder, and every primitive keeps its own albedo."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_12392_gb300 import rcp, scenes  # noqa: E402

pytestmark = pytest.mark.gpu


def _arrays(n_tris, n_spheres):
    sc = scenes.random_soup(n_tris, n_spheres, seed=5)
    return sc.tris.copy(), sc.spheres.copy(), sc.albedo, rcp.make_light(0, (10, 30, 10))


@pytest.mark.parametrize("n_tris,n_spheres", [(1, 0), (0, 1), (2, 3), (7, 5), (1001, 33)])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_non_finite_input_is_refused(n_tris, n_spheres, value):
    for which, at in [(0, 0), (0, -1), (0, 9 * n_tris // 2), (1, 0), (1, -1)]:
        tris, sph, alb, light = _arrays(n_tris, n_spheres)
        target = (tris, sph)[which].reshape(-1)
        if target.size == 0:
            continue
        target[at] = value
        with pytest.raises(rcp.RcpError) as e:
            rcp.rcp_scene_create(tris, sph, alb, light)
        assert e.value.status == rcp.RCP_ERR_ARG and ("vertex", "sphere")[which] in str(e.value)
    tris, sph, alb, light = _arrays(n_tris, n_spheres)
    rcp.rcp_scene_destroy(rcp.rcp_scene_create(tris, sph, alb, light))


def test_each_primitive_keeps_its_albedo():
    sc = scenes.random_soup(301, 40, seed=7)
    sc.albedo[:] = np.random.default_rng(1).uniform(0.1, 0.9, sc.albedo.shape).astype(np.float32)
    g = rcp.rcp_scene_create(sc.tris, sc.spheres, sc.albedo, rcp.make_light(0, (10, 30, 10), 1.0))  # all ambient
    try:
        W, H = 160, 120
        ids = np.empty((H, W), np.int32)
        img = rcp.rcp_render_pass(g, rcp.camera_from(sc.poses[0]), W, H, rcp.make_params(0, 0.0, 1.0), out_prim=ids)
        hit = ids >= 0
        assert len(np.unique(ids[hit])) > 100
        assert np.array_equal(img[..., :3][hit], sc.albedo[ids[hit]])
    finally:
        rcp.rcp_scene_destroy(g)
