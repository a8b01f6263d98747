"""The collapse policy asked for is the one built: on separate objects the
surface-area policy fills its nodes better than the area policy."""
import pytest

pytest.importorskip("torch")

from paper_2312_12392_gb300 import rcp, scenes  # noqa: E402
import gpu_util as U  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [0, 8])
def test_policies_build_different_trees(split):
    sc = scenes.forest_scene(100)
    nodes = {}
    for collapse in (rcp.RCP_COLLAPSE_AREA, rcp.RCP_COLLAPSE_SAH):
        g = U.gpu_scene(sc, collapse, split)
        nodes[collapse] = rcp.rcp_scene_get_info(g).n_nodes
        rcp.rcp_scene_destroy(g)
    assert nodes[rcp.RCP_COLLAPSE_SAH] < 0.9 * nodes[rcp.RCP_COLLAPSE_AREA]
