"""The support rows' chunked placement at its edges: pairs around the head chunks' total of 2,048
per view and one more, a view without pairs between others, one tile row, more tile rows than
the compiled tables hold (288), and views of more than 16 in number (the wider split by view).
Tile lists are in depth order and partition the instances; the rows counted are the rectangles'
rows; the image is that of the same views rendered one by one (same tiles, same lists)."""
import numpy as np
import pytest

from paper_2503_18682_gb300 import scenes
from tests.gpu_util import gpu_render, view_slice
from tests.test_gpu_binning import CULLED, fetch, instance_lists

pytestmark = pytest.mark.gpu


def _case(name):
    cam = scenes.make_camera
    away = scenes.look_at([0.0, 0.0, 8.0], [0.0, 0.0, 12.0])     # sees nothing
    turned = scenes.look_at([0.4, 0.1, -0.5], [0.0, 0.0, 3.0])
    if name == "head_chunks":
        return 2048, [cam(64, 40, 50.0, 50.0)], {}
    if name == "past_head":
        return 2049, [cam(64, 40, 50.0, 50.0), cam(50, 61, 60.0, 60.0, R=turned[0], t=turned[1])], {}
    if name == "empty_view":
        return 3000, [cam(64, 40, 50.0, 50.0), cam(40, 40, 50.0, 50.0, R=away[0], t=away[1]),
                      cam(50, 61, 60.0, 60.0, R=turned[0], t=turned[1])], {}
    if name == "one_row":
        return 700, [cam(90, 7, 50.0, 50.0)], dict(tile_w=8, tile_h=8)
    if name == "tall":
        return 2500, [cam(24, 2400, 300.0, 300.0)], dict(tile_w=8, tile_h=8)
    return 900, [cam(20 + v, 33 + v, 30.0 + v, 31.0, R=turned[0], t=turned[1]) for v in range(19)], {}


@pytest.mark.parametrize("name", ["head_chunks", "past_head", "empty_view", "one_row", "tall", "many_views"])
def test_rows_at_chunk_edges(name):
    n, cams, cfg = _case(name)
    scene = scenes.uniform_scene(n, seed=81)
    r, _, rgb, T, nc = gpu_render(scene, cams, **cfg)
    ctr = r.last_counters
    keys = fetch(r.debug_buffer(0), n * len(cams), np.uint32)
    rects = fetch(r.debug_buffer(1), 2 * n * len(cams), np.uint32).reshape(-1, 2)
    vis = keys != CULLED
    rows = (rects[vis, 1] >> 16).astype(np.int64) - (rects[vis, 0] >> 16) + 1
    assert ctr["n_visible"] == int(vis.sum()) and ctr["n_rows"] == int(rows.sum())
    tiles, pos = instance_lists(r, ctr["n_instances"])
    assert np.all(np.diff(pos)[np.diff(tiles) == 0] > 0)
    for v, c in enumerate(cams):
        _, _, rgb1, T1, nc1 = gpu_render(scene, [c], **cfg)
        sl = view_slice(r, v)
        assert np.array_equal(rgb[sl], rgb1) and np.array_equal(T[sl], T1) and np.array_equal(nc[sl], nc1), v
