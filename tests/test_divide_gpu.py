"""The shared-scale divisions of the sweeps (csrc/divide.cuh) against CUDA's own
division: the same value for every finite operand, zero, infinity and NaN (the
sign of a zero aside)."""
import ctypes
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1905_01330_gb300", "csrc")

SOURCE = r"""
#include <math.h>
#include <stdint.h>
#include "divide.cuh"
using namespace tn;

__device__ uint32_t mix(uint64_t x) {  // splitmix64
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return (uint32_t)((x ^ (x >> 31)) >> 16);
}
// Random sign and mantissa (a quarter of them within four of either end), the
// exponent in [lo, hi].
__device__ float number(uint64_t key, int lo, int hi) {
  const uint32_t a = mix(3 * key), b = mix(3 * key + 1), c = mix(3 * key + 2);
  uint32_t m = a & 0x7FFFFFu;
  if ((c & 3u) == 0u) m = (c & 4u) ? (c >> 8) & 3u : 0x7FFFFFu - ((c >> 8) & 3u);
  const int e = lo + (int)(b % (uint32_t)(hi - lo + 1));
  const float f = ldexpf(1.0f + (float)m * 0x1p-23f, e);
  return (c & 0x40000000u) ? -f : f;
}
__device__ bool same(float a, float b) { return a == b || (isnan(a) && isnan(b)); }

__global__ void check(uint64_t seed, int elo, int ehi, int slo, int shi, unsigned long long* bad) {
  const uint64_t t = seed * 33554432ull + blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  const float special[8] = {0.0f, -0.0f, INFINITY, -INFINITY, NAN, 0x1p-149f, 0x1.fffffep127f, 0x1p-126f};
  // any values, a scale each row, the same in eight neighbouring threads
  float v[4][4], s[4], w[4][4];
  for (int i = 0; i < 4; ++i) {
    s[i] = fabsf(number(64 * (t >> 3) + i, slo, shi));
    if ((t >> 5) % 64 == 9 && mix((t >> 3) + i) % 20u == 0u) s[i] = fabsf(special[mix((t >> 3) + 8 * i) & 7u]);
    for (int j = 0; j < 4; ++j) {
      v[i][j] = number(64 * t + 8 + 4 * i + j, elo, ehi);
      const uint32_t k = mix(977 * t + 4 * i + j);
      if (k % 61u == 0u) v[i][j] = 0.0f;
      if ((t >> 5) % 64 == 7 && k % 97u == 0u) v[i][j] = special[(k >> 8) & 7u];
      w[i][j] = v[i][j];
    }
  }
  divide_rows<false>(w, s);
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 4; ++j)
      if (!same(w[i][j], v[i][j] / s[i])) atomicAdd(bad, 1ull);
  // and none above its scale, eight rows and two
  float v8[8][1], s8[8], v2[2][2], s2[2];
  for (int i = 0; i < 8; ++i) {
    s8[i] = fabsf(number(64 * (t >> 3) + 16 + i, slo, shi));
    v8[i][0] = fminf(fabsf(v[i & 3][i >> 2]), s8[i]);
  }
  for (int i = 0; i < 2; ++i) {
    s2[i] = s8[i + 2];
    for (int j = 0; j < 2; ++j) v2[i][j] = -fminf(fabsf(v[i][j + 2]), s2[i]);
  }
  float w8[8][1], w2[2][2];
  for (int i = 0; i < 8; ++i) w8[i][0] = v8[i][0];
  for (int i = 0; i < 4; ++i) w2[i >> 1][i & 1] = v2[i >> 1][i & 1];
  divide_rows<true>(w8, s8);
  divide_rows<true>(w2, s2);
  for (int i = 0; i < 8; ++i)
    if (!same(w8[i][0], v8[i][0] / s8[i])) atomicAdd(bad, 1ull);
  for (int i = 0; i < 4; ++i)
    if (!same(w2[i >> 1][i & 1], v2[i >> 1][i & 1] / s2[i >> 1])) atomicAdd(bad, 1ull);
  // values up to one scale a warp
  const float top = fabsf(number(77 * (t >> 5) + 5, slo, shi));
  float x[4], y[4];
  for (int j = 0; j < 4; ++j) {
    x[j] = ldexpf(number(64 * t + 40 + j, -44, 0), 0) * top;
    if (!(fabsf(x[j]) <= top)) x[j] = top;
    if (mix(31 * t + j) % 61u == 0u) x[j] = 0.0f;
    y[j] = x[j];
  }
  divide_by_max(y, top);
  for (int j = 0; j < 4; ++j)
    if (!same(y[j], x[j] / top)) atomicAdd(bad + 1, 1ull);
}

extern "C" int run(uint64_t seed, int elo, int ehi, int slo, int shi, unsigned long long* bad) {
  check<<<4096, 256>>>(seed, elo, ehi, slo, shi, bad);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1905_01330_gb300 import build
    d = tmp_path_factory.mktemp("divide")
    src, so = d / "check.cu", d / "check.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-I", CSRC, "-shared", "-Xcompiler", "-fPIC", "-o",
                    str(so), str(src)], check=True, timeout=300)
    h = ctypes.CDLL(str(so))
    h.run.argtypes = [ctypes.c_uint64] + [ctypes.c_int] * 4 + [ctypes.c_void_p]
    return h


@pytest.mark.parametrize("values,scales", [
    ((-20, 4), (-6, 12)),         # a sweep's numbers
    ((-101, -98), (-25, 24)),     # around the least value the correction is used for
    ((97, 101), (-25, 24)),       # and the largest
    ((-40, 40), (-63, -58)), ((-40, 40), (58, 63)), ((-40, 40), (-26, -22)), ((-40, 40), (22, 26)),   # scales likewise
    ((-149, 127), (-149, 127)),   # everything, subnormal numbers too
])
def test_divisions_round_as_cuda_does(lib, values, scales):
    bad = torch.zeros(2, dtype=torch.int64, device="cuda")
    for seed in range(8):  # 32 quotients a thread, 2^20 threads
        assert lib.run(seed, *values, *scales, bad.data_ptr()) == 0
    assert bad.tolist() == [0, 0]
