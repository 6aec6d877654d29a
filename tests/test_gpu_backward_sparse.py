"""Gradients where most primitives have none: the parameter chain rule lists the primitives with a
gradient by chunks of 64 to 512, the more primitives the longer.  A scene among primitives that no
view sees has the same bits as the scene alone (the same sums in the same order), and the others'
gradients are zero."""
import numpy as np
import pytest

from paper_2503_18682_gb300 import scenes
from tests.test_gpu_backward import KEYS, gpu_grads, small_scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("deg,n", [(0, 401), (3, 463), (1, 160001), (2, 320003), (0, 650001)])
def test_unseen_primitives_leave_the_gradients(deg, n):
    sc = small_scene(81 + deg, 400, deg)
    sc["log_scales"][:40, 0] -= 6.0                       # some go through the FP64 kernel
    R1, t1 = scenes.look_at([0.3, -0.2, -0.5], [0, 0, 3.0])
    cams = [scenes.make_camera(83, 61, 70.0, 70.0), scenes.make_camera(37, 29, 30.0, 30.0, R=R1, t=t1)]
    P = sum(c["width"] * c["height"] for c in cams)
    target = np.random.default_rng(9).uniform(0, 1, (P, 3))
    alone, image = gpu_grads(sc, cams, target)
    at = np.sort(np.random.default_rng(n).choice(n, 400, replace=False))
    big = dict(sh_degree=deg)
    for k in KEYS:
        big[k] = np.repeat(sc[k][:1], n, axis=0)
        big[k][at] = sc[k]
    rest = np.ones(n, bool)
    rest[at] = False
    big["means"][rest] = [0.1, 0.2, -40.0]                # behind both cameras
    g, image2 = gpu_grads(big, cams, target)
    assert np.array_equal(image, image2)
    for k in KEYS:
        assert np.abs(alone[k]).max() > 0
        assert np.array_equal(g[k][at], alone[k]), k
        assert not g[k][rest].any(), k


def _replayed(r, nc, tile):
    """Records of all tiles and of the longest one, up to the last composited instance."""
    import torch
    total, longest = 0, 0
    for v, c in enumerate(r.cams):
        im = r.view_image(nc.view(-1, 1), v)[..., 0]
        h, w = -(-c["height"] // tile[1]) * tile[1], -(-c["width"] // tile[0]) * tile[0]
        full = torch.zeros((h, w), dtype=im.dtype, device=im.device)
        full[:c["height"], :c["width"]] = im
        last = full.view(h // tile[1], tile[1], w // tile[0], tile[0]).amax((1, 3))
        total, longest = total + int(last.sum()), max(longest, int(last.max()))
    return total, longest


@pytest.mark.parametrize("tile", [(16, 16), (16, 8), (32, 16), (8, 8)])
def test_split_replay_equals_whole(tile):
    """The replay for few records (up to 3 longest lists per SM) against the one for many: a view
    alone, and with crowded further views whose images have no gradient and so add zeros."""
    import torch
    from paper_2503_18682_gb300 import raygs
    sc = small_scene(91, 3000, 1)
    sc["opacity_logits"][:300] = 9.0                      # clamped opacities
    st = raygs.scene_to_device(sc)
    view, crowd = scenes.make_camera(101, 75, 90.0, 85.0), scenes.make_camera(1920, 1408, 1700.0, 1700.0)
    rng = torch.Generator(device="cuda").manual_seed(5)
    px = view["width"] * view["height"]
    d_rgb, d_T = torch.randn((px, 3), device="cuda", generator=rng), torch.randn(px, device="cuda", generator=rng)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    got = []
    for cams, split in (([view], True), ([view] + 3 * [crowd], False)):
        r = raygs.Renderer(cams, 3000, enable_backward=1, tile_w=tile[0], tile_h=tile[1])
        rgb, T, nc = r.forward(st)
        total, longest = _replayed(r, nc, tile)
        assert (total <= 3 * sms * longest) == split
        full_rgb, full_T = torch.zeros_like(rgb), torch.zeros_like(T)
        full_rgb[:px], full_T[:px] = d_rgb, d_T
        got.append(r.backward(st, T, nc, full_rgb, full_T))
    for k in KEYS:
        a, b = got[0][k], got[1][k]
        assert torch.isfinite(a).all() and a.abs().max() > 0
        assert torch.equal(a, b), k
