"""raygs_render_noalloc where its array leaves no room for what only makes it faster: a batch of 64 views
near the size limit (no head chunks in the row pass), and more than 8,192 tiles (no tile order).  The
images are those of the plan path, bit for bit."""
import numpy as np
import pytest

from paper_2503_18682_gb300 import scenes

pytestmark = pytest.mark.gpu


def _near_limit():
    n = 3757
    scene = scenes.uniform_scene(n, seed=35)
    scene["means"][300:, 2] = -40.0                      # behind every camera
    poses = [scenes.look_at([0.02 * v - 0.6, 0.01 * v, -0.5], [0.0, 0.0, 3.0]) for v in range(64)]
    return scene, [scenes.make_camera(16, 2048, 600.0, 600.0, R=R, t=t) for R, t in poses]


def _many_tiles():
    scene = scenes.uniform_scene(2000, seed=36)
    scene["log_scales"] -= np.float32(1.5)
    return scene, [scenes.make_camera(2050, 1100, 1000.0, 1000.0)]


@pytest.mark.parametrize("case", [_near_limit, _many_tiles])
def test_same_image_without_the_extras(case):
    torch = pytest.importorskip("torch")
    from paper_2503_18682_gb300 import raygs
    scene, cams = case()
    n = scene["means"].shape[0]
    st = raygs.scene_to_device(scene)
    ref = raygs.Renderer(cams, n)
    rgb0, T0, nc0 = ref.forward(st)
    assert int(nc0.max()) > 0
    rgb, T, nc = (torch.full_like(x, -1) for x in (rgb0, T0, nc0))
    assert raygs.raygs_render_noalloc(cams, raygs.make_scene(st), None, rgb, T, nc, check=False) == 0
    assert torch.equal(rgb, rgb0) and torch.equal(T, T0) and torch.equal(nc, nc0)
