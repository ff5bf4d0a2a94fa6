"""The integer implementations of IEEE double operations in ecmc_dev.cuh
(sqrt_rn, div_rn, square_rn) against the compiler's own operations
on the device: every bit equal, over random operands of several exponent
ranges and operands built to sit next to a rounding boundary (squares and
products of short and long mantissas and their neighbours, mantissas of all
ones), and the special values that take the fallback.  f32_trunc against a conversion rounded towards zero."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include "ecmc_dev.cuh"
using namespace ecmc;
__device__ unsigned long long bad[4];
__device__ uint64_t mix(uint64_t x) {
  x ^= x >> 33; x *= 0xff51afd7ed558ccdull; x ^= x >> 33; x *= 0xc4ceb9fe1a85ec53ull;
  return x ^ (x >> 33);
}
__device__ double at(uint64_t e, uint64_t m) { return __longlong_as_double((long long)((e << 52) | (m & 0xFFFFFFFFFFFFFull))); }
__device__ double nudge(double x, int k) { return __longlong_as_double(__double_as_longlong(x) + k); }
__device__ double gen(uint64_t u, int kind) {
  const uint64_t m = u & 0xFFFFFFFFFFFFFull, h = u >> 52;
  switch (kind & 7) {
    case 0: return at(1013 + h % 20, m);
    case 1: return at(540 + h % 960, m);
    case 2: return at(1020 + h % 6, (h & 64) ? ~(m & 0xFF) : (m & 0xFF));
    case 3: { const double s = at(1023, m & ~0x3FFFFFFull); return s * s; }
    case 4: { const double s = at(1023, m); return nudge(s * s, (int)(h % 5) - 2); }
    case 5: return at(1023, m & ~0xFFFull);
    case 6: return at(1022, m | 0xFFFull);
    default: return at(900 + h % 240, m);
  }
}
__device__ bool same(double a, double b) { return __double_as_longlong(a) == __double_as_longlong(b) || (a != a && b != b); }
__device__ void one(double a, double b) {
  if (!same(sqrt(fabs(a)), sqrt_rn(fabs(a)))) atomicAdd(&bad[0], 1ull);
  if (!same(a / b, div_rn(a, b))) atomicAdd(&bad[1], 1ull);
  if (!same(a * a, square_rn(a))) atomicAdd(&bad[2], 1ull);
  if (fabs(a) < 1e38 && (a == 0.0 || fabs(a) > 1e-37) && __double2float_rz(a) != f32_trunc(a)) atomicAdd(&bad[3], 1ull);
}
__global__ void k(uint64_t seed, int n) {
  const uint64_t id = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (int i = 0; i < n; ++i) {
    const uint64_t u = mix(seed + id * 0x9E3779B97F4A7C15ull + i * 0xD1B54A32D192ED03ull), w = mix(u + 77);
    double a = gen(u, (int)(id + i)), b = gen(w, (int)(id / 8 + i));
    if (w >> 63) a = -a;
    if (u >> 63) b = -b;
    one(a, b);
    one(nudge(b * gen(mix(w), i), (int)(u % 3) - 1), b);                // quotients next to a double
  }
}
__global__ void special() {
  const double v[] = {0.0, 1.0, 4.0, 2.0, 0.5, 3.0, 1e-160, 1e160, 1.0 - 0x1p-53, 1.0 + 0x1p-52, 0x1.fffffffffffffp0};
  for (double a : v)
    for (double b : v) {
      if (!same(a / b, div_rn(a, b))) atomicAdd(&bad[1], 1ull);
      if (!same(sqrt(a), sqrt_rn(a))) atomicAdd(&bad[0], 1ull);
      if (!same(a * a, square_rn(a))) atomicAdd(&bad[2], 1ull);
    }
  const double w[] = {-1.0, 1e-310, 1.0 / 0.0, 0.0 / 0.0, 1e308};
  for (double a : w) {
    if (!same(sqrt(a), sqrt_rn(a))) atomicAdd(&bad[0], 1ull);
    if (!same(a / 3.0, div_rn(a, 3.0)) || !same(3.0 / a, div_rn(3.0, a))) atomicAdd(&bad[1], 1ull);
    if (!same(a * a, square_rn(a))) atomicAdd(&bad[2], 1ull);
  }
}
int main() {
  special<<<1, 1>>>();
  for (int r = 0; r < 2; ++r) k<<<2048, 256>>>(12345 + r * 1000003ull, 64);
  unsigned long long h[4];
  if (cudaMemcpyFromSymbol(h, bad, sizeof(h)) != cudaSuccess) return 2;
  std::printf("sqrt %llu div %llu square %llu trunc %llu\n", h[0], h[1], h[2], h[3]);
  return h[0] || h[1] || h[2] || h[3];
}
"""


def test_integer_double_operations_equal_the_hardware(tmp_path):
    nvcc = shutil.which(os.environ.get("NVCC", "nvcc"))
    if nvcc is None:
        pytest.skip("nvcc not found")
    src = tmp_path / "t.cu"
    src.write_text(SRC)
    exe = tmp_path / "t"
    r = subprocess.run([nvcc, "-std=c++17", "-O3", "-fmad=false", "-gencode",
                        "arch=compute_103a,code=sm_103a", "-I",
                        os.path.join(ROOT, "paper_1502_06447_gb300", "csrc"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    if r.returncode != 0:
        pytest.fail(r.stderr[-3000:])
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout + out.stderr
