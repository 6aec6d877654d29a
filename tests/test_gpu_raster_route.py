"""Which of its kernels the rasteriser takes, by tile shape and size of the image: parts of tiles (64
threads) for few tiles, whole tiles for many; the line is lower for 8x8 tiles, where parts are slower from
960x540 on.  The launch is read from a captured graph."""
import ctypes as C

import pytest

from paper_2503_18682_gb300 import scenes

pytestmark = pytest.mark.gpu


class _KernelNode(C.Structure):   # CUDA_KERNEL_NODE_PARAMS
    _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3), ("smem", C.c_uint),
                ("params", C.c_void_p), ("extra", C.c_void_p), ("kern", C.c_void_p), ("ctx", C.c_void_p)]


@pytest.mark.parametrize("tile,size", [((8, 8), (880, 495)), ((8, 8), (960, 540)), ((8, 8), (1280, 720)),
                                       ((16, 8), (1600, 900)), ((16, 8), (1920, 1080))])
@pytest.mark.parametrize("batch_records", [1, 2])
def test_kernel_of_the_rasteriser(tile, size, batch_records):
    import torch
    from paper_2503_18682_gb300 import raygs
    n = 1000
    st = raygs.scene_to_device(scenes.uniform_scene(n, seed=37))
    r = raygs.Renderer([scenes.make_camera(*size, 700.0, 700.0)], n, tile_w=tile[0], tile_h=tile[1],
                       batch_records=batch_records)
    rgb, T, nc = r.forward(st)
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        raygs.raygs_render(r.plan, rgb, T, nc)
    cu, node, count, p = C.CDLL("libcuda.so.1"), C.c_void_p(), C.c_size_t(1), _KernelNode()
    assert cu.cuGraphGetNodes(C.c_void_p(graph.raw_cuda_graph()), C.byref(node), C.byref(count)) == 0
    assert count.value == 1 and cu.cuGraphKernelNodeGetParams_v2(node, C.byref(p)) == 0
    slots = torch.cuda.get_device_properties(0).multi_processor_count * 16 * 256   # pixels of the resident CTAs
    parts = r.num_tiles * tile[0] * tile[1] <= (0.75 if tile == (8, 8) else 2.5) * slots
    whole = 4 * tile[1]
    assert p.block[0] == (64 if parts else whole)
