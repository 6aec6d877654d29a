"""The depth sort of up to 6,144 pairs in one CTA, at its edges: a warp, the CTA's threads, a full
load and one pair past it (the sort in passes); one view, and several sharing the ids."""
import numpy as np
import pytest

from paper_2503_18682_gb300 import scenes
from tests.gpu_util import gpu_render
from tests.test_gpu_binning import CULLED, fetch, instance_lists

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,views", [(31, 1), (512, 1), (513, 1), (2048, 3), (3072, 2), (6143, 1), (6144, 1), (6145, 1)])
def test_order_in_one_cta(n, views):
    scene = scenes.uniform_scene(n, seed=73)
    scene["means"][n // 3:n // 3 + 20] = scene["means"][n // 2]      # exact depth ties
    scene["log_scales"][:5] += 4.0                                    # supports over every tile row
    cams = [scenes.make_camera(70 + 9 * v, 50 + 700 * v, 60.0, 60.0) for v in range(views)]
    r, _, rgb, T, nc = gpu_render(scene, cams)
    keys = fetch(r.debug_buffer(0), n * views, np.uint32)
    vis = np.nonzero(keys != CULLED)[0]
    order = vis[np.argsort(keys[vis], kind="stable")]
    assert r.last_counters["n_visible"] == len(order) > 0
    np.testing.assert_array_equal(fetch(r.debug_buffer(3), len(order), np.uint32), order)
    tiles, pos = instance_lists(r, r.last_counters["n_instances"])
    assert len(tiles) and np.all(np.diff(pos)[np.diff(tiles) == 0] > 0)
    # a view alone has the same image
    v = views - 1
    _, _, rgb1, T1, nc1 = gpu_render(scene, [cams[v]])
    o, px = r.pixel_offsets[v], cams[v]["width"] * cams[v]["height"]
    assert np.array_equal(rgb[o:o + px], rgb1) and np.array_equal(T[o:o + px], T1)
