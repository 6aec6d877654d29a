"""The rasteriser's three ways to cut the image (whole tiles; half tiles with two pixels per
thread; 8x8 blocks with one) give the same bits: a view alone, where its few tiles are taken in
parts, against the same view in a batch large enough for whole tiles."""
import numpy as np
import pytest

from paper_2503_18682_gb300 import scenes
from tests.gpu_util import gpu_render, view_slice

pytestmark = pytest.mark.gpu


def _same(scene, alone, batch, **cfg):
    r, _, rgb, T, nc = gpu_render(scene, batch, **cfg)
    _, _, rgb1, T1, nc1 = gpu_render(scene, [alone], **cfg)
    sl = view_slice(r, 0)
    assert np.array_equal(rgb[sl], rgb1) and np.array_equal(T[sl], T1) and np.array_equal(nc[sl], nc1)
    assert nc1.max() > 0


@pytest.mark.parametrize("batch_records", [1, 2])
@pytest.mark.parametrize("tile", [(16, 16), (16, 8), (32, 16), (8, 8)])
@pytest.mark.parametrize("divergence", [0, 1])
def test_parts_equal_whole_tiles(tile, batch_records, divergence):
    cfg = dict(tile_w=tile[0], tile_h=tile[1], batch_records=batch_records, divergence=divergence)
    # blocks of one pixel per thread: 110 ragged tiles alone, 7,040 in the batch
    scene = scenes.uniform_scene(2500, seed=91)
    scene["log_scales"][:200, 0] -= 5.0                 # slivers: the conservative test's hard case
    small = scenes.make_camera(171, 149, 150.0, 140.0)
    _same(scene, small, [small] * 64, **cfg)
    # two pixels per thread: 1,200 tiles with long lists alone, 9,600 in the batch
    scene = scenes.uniform_scene(30000, seed=92)
    scene["log_scales"][:2000, 1] -= 5.0
    view = scenes.make_camera(633, 478, 420.0, 430.0)
    _same(scene, view, [view] * 8, **cfg)


@pytest.mark.parametrize("tile", [(16, 16), (16, 8), (32, 16), (8, 8)])
def test_exact_antialiasing_parts(tile):
    """The exact anti-aliasing's region shapes (8x8 blocks with one or two pixels per thread, larger
    regions with two) give the same bits."""
    cfg = dict(tile_w=tile[0], tile_h=tile[1])
    scene = scenes.uniform_scene(2500, seed=93)
    small = scenes.make_camera(171, 149, 150.0, 140.0, mip="exact")
    _same(scene, small, [small] * 30, **cfg)            # alone one pixel; 3,300 tiles: two in blocks
    _same(scene, small, [small] * 64, **cfg)            # 7,040 tiles: larger regions
