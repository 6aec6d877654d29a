"""Views at the ends of the binning's range: wider than 526 and 2,047 tile columns (the instance lists' two
smaller shapes), where each tile's list is in depth order, no dropped tile holds a pixel of the support and the
image keeps oracle parity; and taller than 288 tile rows with the backward (the row pass's run-time table
beside the partial sums), against autograd through the dense FP64 reference."""
import numpy as np
import pytest

from paper_2503_18682_gb300 import scenes
from tests.gpu_util import assert_parity, compare, gpu_render, sample_pixels
from tests.test_gpu_backward import assert_close_grads, gpu_grads, ref_grads, small_scene
from tests.test_gpu_binning import assert_dropped_tiles_miss_support, fetch, instance_lists

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,height", [(4208, 24), (4216, 24), (16376, 16), (17001, 8)])
def test_wide_views(oracle_lib, width, height):
    n = 1500
    sc = scenes.uniform_scene(n, seed=42)
    sc["means"][:, 0] *= np.float32(width / 1000)
    sc["means"][:, 1] *= np.float32(0.02)
    sc["log_scales"][:200, 0] += np.float32(3.0)          # some long ones
    cam = scenes.make_camera(width, height, 1000.0, 1000.0)
    r, _, rgb, T, nc = gpu_render(sc, [cam], tile_w=8, tile_h=8)
    tiles, pos = instance_lists(r, r.last_counters["n_instances"])
    assert len(np.unique(tiles)) > r.num_tiles // 2
    assert np.all(np.diff(pos)[np.diff(tiles) == 0] > 0)
    order = fetch(r.debug_buffer(3), r.last_counters["n_visible"], np.uint32)
    assert_dropped_tiles_miss_support(oracle_lib, sc, [cam], r, n, (8, 8), {int(p) for p in order[::60]})
    pix, idx = sample_pixels(cam, 1500, seed=5)
    assert_parity(compare(rgb[idx], T[idx], oracle_lib.render(sc, cam, pixels=pix)))


def test_backward_of_a_tall_view():
    sc = small_scene(95, 220, 1)
    sc["means"][:, 0] *= np.float32(0.01)
    sc["means"][:, 1] *= np.float32(7.0)
    cam = scenes.make_camera(7, 2390, 480.0, 500.0)
    target = np.random.default_rng(10).uniform(0, 1, (7 * 2390, 3))
    g, image = gpu_grads(sc, [cam], target, tile_w=8, tile_h=8)
    assert image.max() > 0
    assert_close_grads(g, ref_grads(sc, [cam], target))
