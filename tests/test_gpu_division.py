"""The backward's division (an approximate reciprocal, one Newton step and one residual correction) against
CUDA's: over the ranges of its divisors and dividends at most one ulp off, in fewer than one of 2^20 cases (the
reciprocal alone: 2^19); and infinite gradients from the caller stay infinite, as with the division
operator."""
import ctypes as C

import numpy as np
import pytest

from paper_2503_18682_gb300 import scenes
from tests.gpu_probe import compile_probe

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "raster_math.cuh"
using namespace raygs;
__device__ uint32_t mix(uint32_t x) {
  x ^= x >> 16; x *= 0x7feb352dU; x ^= x >> 15; x *= 0x846ca68bU; x ^= x >> 16;
  return x;
}
// random mantissa, exponent in [lo, hi)
__device__ float draw(uint32_t seed, int lo, int hi) {
  const uint32_t a = mix(seed), b = mix(seed ^ 0x9e3779b9U);
  return __uint_as_float((uint32_t(127 + lo + int(b % uint32_t(hi - lo))) << 23) | (a & 0x7fffffU));
}
// out: {mismatches, largest difference in ulp} of 1 / x and of a / x
__global__ void check(uint32_t n, int xlo, int xhi, int alo, int ahi, unsigned *out) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float x = draw(4 * i + 1, xlo, xhi), a = draw(4 * i + 2, alo, ahi) * (i & 1 ? -1.f : 1.f);
    const float r = rcp_newton(x), q = div_newton(a, x, r), any = div_newton_any(a, x, r);
    const int dr = abs(__float_as_int(r) - __float_as_int(1.f / x)), dq = abs(__float_as_int(q) - __float_as_int(a / x));
    if (dr) atomicAdd(out, 1u), atomicMax(out + 1, unsigned(dr));
    if (dq) atomicAdd(out + 2, 1u), atomicMax(out + 3, unsigned(dq));
    if (__float_as_int(any) != __float_as_int(q)) atomicAdd(out + 4, 1u);
  }
}
__global__ void pairs(const float *a, const float *x, int n, float *out) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    out[2 * i] = div_newton_any(a[i], x[i], rcp_newton(x[i]));
    out[2 * i + 1] = a[i] / x[i];
  }
}
extern "C" int run_check(uint32_t n, int xlo, int xhi, int alo, int ahi, unsigned *out) {
  check<<<1024, 256>>>(n, xlo, xhi, alo, ahi, out);
  return int(cudaDeviceSynchronize());
}
extern "C" int run_pairs(const float *a, const float *x, int n, float *out) {
  pairs<<<1, 256>>>(a, x, n, out);
  return int(cudaDeviceSynchronize());
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    torch = pytest.importorskip("torch")
    torch.cuda.init()
    return compile_probe(SOURCE, str(tmp_path_factory.mktemp("division")))


# 1 - omega (down to the largest accepted alpha_max) under T and under the loss gradients; D's denominator
@pytest.mark.parametrize("x,a", [((-24, 0), (-14, 0)), ((-24, 0), (-60, 60)), ((-100, 100), (-10, 20))])
def test_division_is_within_its_bound(probe, x, a):
    import torch
    n = 1 << 27
    out = torch.zeros(5, dtype=torch.int32, device="cuda")
    assert probe.run_check(C.c_uint32(n), x[0], x[1], a[0], a[1], C.c_void_p(out.data_ptr())) == 0
    rcp_off, rcp_ulp, div_off, div_ulp, any_off = out.tolist()
    assert rcp_ulp <= 1 and rcp_off <= n >> 19
    assert div_ulp <= 1 and div_off <= n >> 20
    assert any_off == 0


def test_division_of_any_dividend(probe):
    import torch
    inf, big = float("inf"), float(np.finfo(np.float32).max)
    a = np.array([inf, -inf, float("nan"), 0.0, -0.0, big, -big, big / 8, -3e38, 1e-30], np.float32)
    x = np.array([1.0, 0.75, 0.01, 2.0 ** -24], np.float32)
    aa, xx = (torch.tensor(v.ravel().copy(), device="cuda") for v in np.meshgrid(a, x))
    out = torch.empty((aa.numel(), 2), device="cuda")
    assert probe.run_pairs(C.c_void_p(aa.data_ptr()), C.c_void_p(xx.data_ptr()), aa.numel(), C.c_void_p(out.data_ptr())) == 0
    got, want = out[:, 0].cpu().numpy(), out[:, 1].cpu().numpy()
    np.testing.assert_array_equal(got, want)


@pytest.mark.parametrize("crowd", [0, 3])
def test_infinite_gradient_of_the_transmittance(crowd):
    """dL/dT = +-inf at one pixel: the opacities of the primitives composited there get -+inf, not NaN."""
    import torch
    from paper_2503_18682_gb300 import raygs
    n = 3000
    st = raygs.scene_to_device(scenes.uniform_scene(n, seed=38))
    far = scenes.make_camera(1920, 1408, 1700.0, 1700.0)        # more to replay: the whole-tile replay
    r = raygs.Renderer([scenes.make_camera(64, 48, 60.0, 60.0)] + crowd * [far], n, enable_backward=1)
    rgb, T, nc = r.forward(st)
    at = int(nc[:64 * 48].argmax())
    for sign in (1.0, -1.0):
        d_T = torch.zeros_like(T)
        d_T[at] = sign * float("inf")
        g = r.backward(st, T, nc, torch.zeros_like(rgb), d_T)["opacity_logits"]
        hit = ~torch.isfinite(g)
        assert int(hit.sum()) > 0 and bool((g[hit] == -sign * float("inf")).all())
