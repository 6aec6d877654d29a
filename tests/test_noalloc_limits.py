"""What raygs_render_noalloc takes: the largest batches of 64 views that fit its array, and its instance
capacity, never fall below what callers have been able to rely on (133 bytes per (primitive, view), 12
per tile, 36 per tile row and tile column at most, 45 per instance).  Host only."""
import ctypes as C

import pytest

from paper_2503_18682_gb300 import scenes

ARRAY = 32 << 20


@pytest.fixture(scope="module")
def capacity():
    from paper_2503_18682_gb300 import build, raygs
    build.build()
    fn = raygs.lib().raygs_debug_noalloc_capacity
    fn.restype = C.c_int64

    def of(cams, n, tile=(16, 16)):
        cfg = raygs.make_config(tile_w=tile[0], tile_h=tile[1])
        return fn(raygs.make_cameras(cams), len(cams), C.c_int64(n), C.byref(cfg), 152)
    return of


@pytest.mark.parametrize("w,h,n", [(640, 480, 3643), (1024, 1024, 3290), (1920, 1080, 2800), (16, 2048, 3757)])
def test_largest_batches_of_64_views_are_taken(capacity, w, h, n):
    assert capacity([scenes.make_camera(w, h, 50.0, 50.0)] * 64, n) > 0


def test_refuses_what_cannot_fit(capacity):
    assert capacity([scenes.make_camera(32, 32, 32.0, 32.0)], 400_000) == 0


@pytest.mark.parametrize("views,w,h,tile", [(1, 64, 64, (16, 16)), (1, 2064, 2208, (8, 8)), (2, 640, 480, (16, 8)),
                                            (3, 32768, 8, (8, 8)), (17, 300, 200, (32, 16)), (64, 8, 4000, (8, 8))])
@pytest.mark.parametrize("fill", [0.0, 0.3, 0.8, 0.95])
def test_capacity(capacity, views, w, h, tile, fill):
    """The capacity left by a batch that fills the given part of the array."""
    tx, ty = -(-w // tile[0]), -(-h // tile[1])
    fixed = 1_300_000 + views * (160 + ty * (20 + 4 * tx) + 12 * tx * ty)   # sort tables, views, rows, tiles
    n = int(fill * (ARRAY - fixed) / (133 * views))
    left = ARRAY - fixed - 133 * views * n
    want = int(left / (45 + 4 * tx / 8192)) - 4096
    assert capacity([scenes.make_camera(w, h, 50.0, 50.0)] * views, n, tile) >= max(want, 1)
