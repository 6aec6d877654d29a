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
