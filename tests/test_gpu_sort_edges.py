"""The depth sort at the edges of its launch rules: one item, a full tile of 2,048 and one more,
the largest grid whose downsweep reads every CTA's counts itself (16 tiles) and one item past it."""
import numpy as np
import pytest

from paper_2503_18682_gb300 import scenes
from tests.gpu_util import gpu_render
from tests.test_gpu_binning import CULLED, fetch, instance_lists

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2048, 2049, 16 * 2048, 16 * 2048 + 1])
def test_depth_order_at_grid_edges(n):
    scene = scenes.uniform_scene(n, seed=71)
    scene["means"][n // 3:n // 3 + 20] = scene["means"][n // 2]      # exact depth ties
    r, _, rgb, T, nc = gpu_render(scene, [scenes.make_camera(70, 50, 60.0, 60.0)])
    keys = fetch(r.debug_buffer(0), n, np.uint32)
    vis = np.nonzero(keys != CULLED)[0]
    order = vis[np.argsort(keys[vis], kind="stable")]
    assert r.last_counters["n_visible"] == len(order)
    if len(order):
        np.testing.assert_array_equal(fetch(r.debug_buffer(3), len(order), np.uint32), order)
    tiles, pos = instance_lists(r, r.last_counters["n_instances"])
    assert np.all(np.diff(pos)[np.diff(tiles) == 0] > 0)
