"""The rasterisers' conservative box test on 8x8 blocks of a 32 pixel wide tile: no record that a pixel of the
block composites is dropped.  Slivers and cone edges are drawn so that a pixel of the block lies within
rounding of the support's border, in the columns that the pixel evaluation reaches after the most steps."""
import ctypes as C

import pytest

from tests.gpu_probe import compile_probe

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "raster_math.cuh"
using namespace raygs;
__device__ uint32_t mix(uint32_t x) {
  x ^= x >> 16; x *= 0x7feb352dU; x ^= x >> 15; x *= 0x846ca68bU; x ^= x >> 16;
  return x;
}
struct Draw {
  uint32_t s;
  __device__ double u(double a, double b) { s += 0x9e3779b9U; return a + (b - a) * (mix(s) * (1.0 / 4294967296.0)); }
  __device__ double p10(double a, double b) { return exp10(u(a, b)); }
};
template <int COL>
__device__ bool any_hit(const float4 &A, const float4 &B, int row) {
  float q[1], r[1], y0[1], y1[1], y2[1];
  for (int i = 0; i < 32; ++i)
    if (eval_pixels<1, COL>(A, B, float(i & 3), float(row + (i >> 2)), 4.f, q, r, y0, y1, y2)) return true;
  return false;
}
// out: records that a pixel composites, and those of them that the box test drops
template <int COL>
__global__ void check(uint32_t seed, uint32_t n, unsigned *out) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    Draw d{mix(seed + i)};
    const int row = i & 1 ? 8 : 0;
    float4 A, B;
    if (i & 2) {  // a sliver, its border at a pixel of the block
      const double th = d.u(-0.4, 0.4), w = d.p10(-7, -0.5), len = d.p10(0, 3), along = d.u(-5, 5);
      const double off = w * (1 + d.u(-1, 1) * d.p10(-6, -3)), nx = cos(th), ny = sin(th);
      const double side = i & 4 ? 1.0 : -1.0;
      const double ux = 4 * COL + int(d.u(0, 4)) - side * nx * off + ny * along, uy = row + int(d.u(0, 8)) - side * ny * off - nx * along;
      A = make_float4(float(-ux), float(-uy), float(nx / w), float(ny / w));
      B = make_float4(float(-ny / len), float(nx / len), i & 8 ? float(d.u(-0.01, 0.01)) : 0.f, i & 16 ? float(d.u(-0.01, 0.01)) : 0.f);
    } else {      // a cone whose y2 vanishes beside the block's first column
      const double h = d.p10(0.1, 4), e = d.p10(-6, -1), t = (1 - e) / h;
      A = make_float4(float(t - 4 * COL), float(-row - d.u(-20, 20)), float((1 - h * t) / t * (1 + d.u(-1, 1) * d.p10(-6, -2))), 0.f);
      B = make_float4(0.f, 0.f, float(-h), 0.f);
    }
    if (!any_hit<COL>(A, B, row)) continue;
    atomicAdd(out, 1u);
    if (!box_may_hit(A, B, 4.f * COL + 1.5f, row + 3.5f, 1.5f, 3.5f)) atomicAdd(out + 1, 1u);
  }
}
extern "C" int run(int col, uint32_t seed, uint32_t n, unsigned *out) {
  switch (col) {
    case 0: check<0><<<1024, 128>>>(seed, n, out); break;
    case 3: check<3><<<1024, 128>>>(seed, n, out); break;
    case 5: check<5><<<1024, 128>>>(seed, n, out); break;
    default: check<7><<<1024, 128>>>(seed, n, out); break;
  }
  return int(cudaDeviceSynchronize());
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    torch = pytest.importorskip("torch")
    torch.cuda.init()
    return compile_probe(SOURCE, str(tmp_path_factory.mktemp("box")))


@pytest.mark.parametrize("col", [0, 3, 5, 7])
def test_box_keeps_every_composited_record(probe, col):
    import torch
    n = 1 << 25
    out = torch.zeros(2, dtype=torch.int32, device="cuda")
    assert probe.run(col, C.c_uint32(17 + col), C.c_uint32(n), C.c_void_p(out.data_ptr())) == 0
    hits, dropped = out.tolist()
    assert hits > n // 8 and dropped == 0
