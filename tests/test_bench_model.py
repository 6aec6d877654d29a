"""The benchmark's account of a pass: bytes of the binning kernels, term by term, and kernels per pass."""
import os
import sys

import pytest

from paper_2503_18682_gb300 import scenes

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_bytes_of_a_binning_pass():
    ctr = dict(n_visible=1000, n_rows=3000, n_rows_kept=2500, n_instances=9000)
    rows, lists = 4 * 1000 + 8 * 1000 + 32 * 1000 + 8 * 3000, 2 * 8 * 3000 + 4 * 9000
    sort = 2 * 4 * 9000 + 2 * 1000 + 8 * 1000 + 3 * (4 + 16) * 1000
    assert bench.binning_pass_bytes(ctr, 9000, 1) == sort + rows + lists
    # several views: the split (keys read twice, values once; three words written) and the positions
    assert bench.binning_pass_bytes(ctr, 9000, 4) == sort + rows + lists + (12 + 12) * 1000 + 4 * 1000
    one_cta = 4 * 6000 + 2 * 1000 + 8 * 1000
    assert bench.binning_pass_bytes(ctr, 6000, 1) == one_cta + rows + lists
    # without the row sort that the yardstick counts
    big = dict(n_visible=18_400_000, n_rows=61_000_000, n_rows_kept=54_000_000, n_instances=206_700_000)
    assert bench.binning_pass_bytes(big, 48_000_000, 16) < bench.binning_bytes(big, 48_000_000)


@pytest.mark.gpu
@pytest.mark.parametrize("n,views", [(1000, 1), (6144, 1), (6145, 1), (3000, 2), (4000, 9), (33000, 1)])
def test_launches_of_a_pass(n, views):
    import ctypes as C
    import torch
    from paper_2503_18682_gb300 import raygs
    st = raygs.scene_to_device(scenes.uniform_scene(n, seed=39))
    r = raygs.Renderer([scenes.make_camera(64, 48, 60.0, 60.0)] * views, n)
    out = r.forward(st)
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        r.forward(st, *out, check=False)
    nodes = C.c_size_t(0)
    assert C.CDLL("libcuda.so.1").cuGraphGetNodes(C.c_void_p(graph.raw_cuda_graph()), None, C.byref(nodes)) == 0
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert nodes.value - 1 == bench.launches_per_pass(n * views, views, sms)   # one clear
