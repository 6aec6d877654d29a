"""Views whose tiles' lists are nearly as long as the longest (large primitives) or empty: the rasteriser takes them
in their own order with the most pixels per thread, also where it takes few tiles in parts.  The bits are
those of the same view in a batch of many, or of a plan that keeps no classes (the allocation-free call)."""
import numpy as np
import pytest

from paper_2503_18682_gb300 import scenes
from tests.gpu_util import gpu_render, view_slice
from tests.test_gpu_binning import fetch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch_records", [1, 2])
@pytest.mark.parametrize("divergence", [0, 1])
@pytest.mark.parametrize("tile", [(16, 16), (16, 8), (32, 16), (8, 8)])
def test_even_lists_alone_and_in_a_batch(tile, divergence, batch_records):
    import torch
    cfg = dict(tile_w=tile[0], tile_h=tile[1], divergence=divergence, batch_records=batch_records)
    scene = scenes.uniform_scene(600, seed=94)
    scene["log_scales"] += np.float32(2.0)
    view = scenes.make_camera(1267, 713, 1000.0, 1000.0)
    r1, _, rgb1, T1, nc1 = gpu_render(scene, [view], **cfg)
    ranges = fetch(r1.debug_buffer(6), 2 * r1.num_tiles, np.uint32).reshape(-1, 2).astype(np.int64)
    lists = ranges[:, 1] - ranges[:, 0]
    slots = 18 * torch.cuda.get_device_properties(0).multi_processor_count
    assert 3 * lists.sum() >= lists.max() * r1.num_tiles                       # taken in their own order
    assert tile == (8, 8) or 10 * tile[0] * tile[1] * lists.sum() >= 4 * 256 * slots * lists.max()
    r, _, rgb, T, nc = gpu_render(scene, [view] * 8, **cfg)
    for v in (0, 7):
        sl = view_slice(r, v)
        assert np.array_equal(rgb[sl], rgb1) and np.array_equal(T[sl], T1) and np.array_equal(nc[sl], nc1)
    assert nc1.max() > 0


@pytest.mark.parametrize("tile", [(16, 16), (32, 16)])
def test_one_long_list_among_empty_ones(tile):
    """All primitives in a corner, and none at all: the other end of the rule."""
    cfg = dict(tile_w=tile[0], tile_h=tile[1])
    scene = scenes.uniform_scene(800, seed=95)
    scene["means"][:, :2] *= np.float32(0.02)
    view = scenes.make_camera(1267, 713, 1000.0, 1000.0, 40.0, 30.0)
    _, _, rgb1, T1, nc1 = gpu_render(scene, [view], **cfg)
    r, _, rgb, T, nc = gpu_render(scene, [view] * 8, **cfg)
    sl = view_slice(r, 3)
    assert np.array_equal(rgb[sl], rgb1) and np.array_equal(T[sl], T1) and np.array_equal(nc[sl], nc1)
    scene["means"][:, 2] = -40.0
    _, _, rgb, T, nc = gpu_render(scene, [view], **cfg)
    assert not rgb.any() and (T == 1).all() and not nc.any()
