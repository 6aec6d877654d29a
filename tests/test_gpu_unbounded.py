"""Many primitives whose support is not a bounded ellipse: all of their rows are bounded as long as the rows
fit the capacity.  A capacity that just holds the rows and instances of a roomy plan gives the same
instances, the same lists and no overflow; below it, the counters are the same from call to call."""
import numpy as np
import pytest

from paper_2503_18682_gb300 import scenes
from tests.gpu_util import gpu_render
from tests.test_gpu_binning import CULLED, fetch, instance_lists

pytestmark = pytest.mark.gpu


def _scene(n):
    rng = np.random.default_rng(71)
    sc = scenes.uniform_scene(n, seed=71)
    sc["means"] = rng.uniform([-0.3, -0.6, 0.03], [0.3, 0.6, 0.3], (n, 3)).astype(np.float32)
    sc["log_scales"] = rng.uniform(np.log(0.03), np.log(0.3), (n, 3)).astype(np.float32)
    sc["log_scales"][:n // 4, 0] -= 8.0                  # some of them go through the FP64 vertex stage
    return sc


@pytest.mark.parametrize("backward", [0, 1])
def test_exact_capacity_is_enough(backward):
    from paper_2503_18682_gb300 import raygs
    n, cams = 1500, [scenes.make_camera(64, 800, 300.0, 300.0), scenes.make_camera(61, 640, 250.0, 250.0)]
    sc = _scene(n)
    cfg = dict(tile_w=8, tile_h=8, enable_backward=backward)
    r, st, rgb, T, nc = gpu_render(sc, cams, capacity=4_000_000, **cfg)
    ctr = dict(r.last_counters)
    tiles, pos = instance_lists(r, ctr["n_instances"])
    keys = fetch(r.debug_buffer(0), n * 2, np.uint32)
    ell = fetch(r.debug_buffer(7), 8 * n * 2, np.uint32).reshape(-1, 8)
    unbounded = (keys != CULLED) & ~(ell[:, 4].view(np.float32) > 0)
    rows = int(((ell[unbounded, 1] >> 16).astype(np.int64) - (ell[unbounded, 0] >> 16) + 1).sum())
    need = max(ctr["n_rows"], ctr["n_instances"])
    assert rows > need // 8 + 1024 and unbounded[:n].sum() > 100 and ctr["n_instances"] < 8 * ctr["n_rows"]

    tight = raygs.Renderer(cams, n, capacity=need, **cfg)
    for _ in range(2):
        out = tight.forward(st, check=False)
        got = raygs.raygs_read_counters(tight.plan)
        assert not got["overflow"]
        assert {k: got[k] for k in ctr if k != "capacity"} == {k: ctr[k] for k in ctr if k != "capacity"}
        t2, p2 = instance_lists(tight, ctr["n_instances"])
        assert np.array_equal(t2, tiles) and np.array_equal(p2, pos)
        for a, b in zip(out, (rgb, T, nc)):
            assert np.array_equal(a.cpu().numpy(), b)

    low = raygs.Renderer(cams, n, capacity=ctr["n_rows"] // 2, **cfg)
    seen = set()
    for _ in range(4):
        low.forward(st, check=False)
        got = raygs.raygs_read_counters(low.plan)
        assert got["overflow"] and got["n_instances"] >= ctr["n_rows"]
        seen.add(tuple(sorted(got.items())))
    assert len(seen) == 1


def test_binning_twice_after_one_vertex_stage():
    """The binning of a plan can be repeated: what it reads of the vertex stage stays."""
    from paper_2503_18682_gb300 import raygs
    sc, cams = _scene(700), [scenes.make_camera(1200, 48, 300.0, 300.0)]
    r, st, rgb, T, nc = gpu_render(sc, cams)
    ctr = dict(r.last_counters)
    tiles, pos = instance_lists(r, ctr["n_instances"])
    for _ in range(2):
        raygs.raygs_bin_sort(r.plan)
        assert raygs.raygs_read_counters(r.plan) == ctr
        t2, p2 = instance_lists(r, ctr["n_instances"])
        assert np.array_equal(t2, tiles) and np.array_equal(p2, pos)
    out = r.alloc_outputs()
    raygs.raygs_render(r.plan, *out)
    assert np.array_equal(out[0].cpu().numpy().astype(np.float64), rgb)
