"""The backward of few tiles: up to three per SM go to the split replay without a plan of the lists, and no
gradient buffer is cleared by a launch of its own.  The gradients are the same bits as those of the same
view beside further tiles, where the plan decides; a pass is five launches."""
import ctypes as C

import numpy as np
import pytest

from paper_2503_18682_gb300 import scenes
from tests.test_gpu_backward import KEYS, small_scene

pytestmark = pytest.mark.gpu


def _grads(sc, cams, px, d_rgb, d_T, **cfg):
    import torch
    from paper_2503_18682_gb300 import raygs
    st = raygs.scene_to_device(sc)
    r = raygs.Renderer(cams, sc["means"].shape[0], enable_backward=1, **cfg)
    rgb, T, nc = r.forward(st)
    full_rgb, full_T = torch.zeros_like(rgb), torch.zeros_like(T)
    full_rgb[:px], full_T[:px] = d_rgb, d_T
    return r, r.backward(st, T, nc, full_rgb, full_T)


@pytest.mark.parametrize("tile", [(16, 16), (16, 8), (32, 16), (8, 8)])
def test_same_bits_with_and_without_a_plan(tile):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sc = small_scene(92, 2500, 1)
    sc["opacity_logits"][:300] = 9.0
    cam = scenes.make_camera(tile[0] * sms // 2 - 3, 6 * tile[1] - 1, 90.0, 60.0)   # three tiles per SM
    px = cam["width"] * cam["height"]
    rng = torch.Generator(device="cuda").manual_seed(6)
    d_rgb, d_T = torch.randn((px, 3), device="cuda", generator=rng), torch.randn(px, device="cuda", generator=rng)
    cfg = dict(tile_w=tile[0], tile_h=tile[1])
    ra, a = _grads(sc, [cam], px, d_rgb, d_T, **cfg)
    rb, b = _grads(sc, [cam, scenes.make_camera(5, 5, 60.0, 60.0)], px, d_rgb, d_T, **cfg)
    assert ra.num_tiles == 3 * sms and rb.num_tiles == 3 * sms + 1
    for k in KEYS:
        assert torch.isfinite(a[k]).all() and a[k].abs().max() > 0
        assert torch.equal(a[k], b[k]), k


def test_launches_of_a_small_backward():
    import torch
    from paper_2503_18682_gb300 import raygs
    sc = small_scene(93, 400, 0)
    st = raygs.scene_to_device(sc)
    r = raygs.Renderer([scenes.make_camera(64, 64, 50.0, 50.0)], 400, enable_backward=1)
    rgb, T, nc = r.forward(st)
    d_rgb = torch.ones_like(rgb)
    want = r.backward(st, T, nc, d_rgb)
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        got = r.backward(st, T, nc, d_rgb)
    nodes = C.c_size_t(0)
    assert C.CDLL("libcuda.so.1").cuGraphGetNodes(C.c_void_p(graph.raw_cuda_graph()), None, C.byref(nodes)) == 0
    assert nodes.value == 5    # one clear; replay, pair sums, parameters, FP64 parameters
    graph.replay()
    for k in KEYS:
        assert np.array_equal(got[k].cpu().numpy(), want[k].cpu().numpy()), k
