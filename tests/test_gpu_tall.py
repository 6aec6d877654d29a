"""Views of thousands of tile rows (the row pass's run-time table, whose cursors are fetched as rows are met): a
few primitives near the camera that cover most of the height among many small ones, in a single view, beside a
low one, and with pairs on both sides of the head chunks.  The rows counted are the rectangles' rows, each
tile's list is in depth order, and the image keeps oracle parity; the backward's numbering gives the
gradients of the same view in larger tiles."""
import numpy as np
import pytest

from paper_2503_18682_gb300 import scenes
from tests.gpu_util import assert_parity, compare, gpu_render, sample_pixels, view_slice
from tests.test_gpu_backward import KEYS
from tests.test_gpu_binning import CULLED, fetch, instance_lists

pytestmark = pytest.mark.gpu


def _scene(n, seed):
    rng = np.random.default_rng(seed)
    sc = scenes.uniform_scene(n, seed=seed)
    sc["means"] = np.stack([rng.uniform(-0.01, 0.01, n), rng.uniform(-2.0, 2.0, n), rng.uniform(1.0, 3.0, n)],
                           axis=1).astype(np.float32)
    sc["log_scales"] = rng.uniform(np.log(0.003), np.log(0.02), (n, 3)).astype(np.float32)
    near = slice(0, 12)
    sc["means"][near, 2] = rng.uniform(0.8, 1.0, 12)
    sc["log_scales"][near, 1] = np.log(1.5)
    sc["opacity_logits"][near] = -2.0
    return sc


@pytest.mark.parametrize("n,sizes", [(700, [(23, 2313)]), (2049, [(24, 8200)]), (5000, [(40, 32768)]),
                                     (3000, [(33, 4100), (50, 60), (16, 12000)])])
def test_tall_views(oracle_lib, n, sizes):
    sc = _scene(n, 43)
    cams = [scenes.make_camera(w, h, 0.4 * max(h, 400), 0.4 * max(h, 400)) for w, h in sizes]
    r, _, rgb, T, nc = gpu_render(sc, cams, tile_w=8, tile_h=8)
    keys = fetch(r.debug_buffer(0), n * len(cams), np.uint32)
    rects = fetch(r.debug_buffer(1), 2 * n * len(cams), np.uint32).reshape(-1, 2)
    rows = (rects[:, 1] >> 16).astype(np.int64) - (rects[:, 0] >> 16) + 1
    assert r.last_counters["n_rows"] == int(rows[keys != CULLED].sum())
    assert rows[keys != CULLED].max() > 256
    tiles, pos = instance_lists(r, r.last_counters["n_instances"])
    assert np.all(np.diff(pos)[np.diff(tiles) == 0] > 0)
    for v, cam in enumerate(cams):
        sl = view_slice(r, v)
        pix, idx = sample_pixels(cam, 800, seed=v)
        assert_parity(compare(rgb[sl][idx], T[sl][idx], oracle_lib.render(sc, cam, pixels=pix)))


def test_gradients_of_a_tall_view_in_small_and_large_tiles():
    import torch
    from paper_2503_18682_gb300 import raygs
    sc = _scene(2500, 44)
    st = raygs.scene_to_device(sc)
    cam = scenes.make_camera(24, 6000, 2400.0, 2400.0)
    got = []
    for tile in ((8, 8), (32, 16)):
        r = raygs.Renderer([cam], 2500, enable_backward=1, tile_w=tile[0], tile_h=tile[1])
        rgb, T, nc = r.forward(st)
        g = torch.Generator(device="cuda").manual_seed(8)
        got.append(r.backward(st, T, nc, torch.randn(rgb.shape, device="cuda", generator=g), None))
    for k in KEYS:
        a, b = got[0][k].double(), got[1][k].double()
        assert torch.isfinite(a).all() and b.abs().max() > 0
        assert ((a - b).abs() <= 2e-3 * b.abs().max() + 3e-3 * b.abs()).all(), k   # the tile shapes' tolerance
