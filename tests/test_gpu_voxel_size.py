"""The voxel size in pairs of floats (leaf_voxel_size) against the definition in FP64
(leaf_voxel_size_fp64), bit for bit: extents of all exponents, flat leaves (floored at
delta), perfect cubes, counts up to and beyond the range of exact floats."""

import subprocess

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include "gd_leaf_kernel.cuh"
#include <cstdio>
#include <cstdlib>
using namespace gd;
__device__ uint32_t rnd(unsigned long long &s) {  // a linear congruential step, its high bits
  s = s * 6364136223846793005ull + 1442695040888963407ull;
  return (uint32_t)(s >> 32);
}
__global__ void k_compare(int mode, unsigned long long *bad) {
  unsigned long long s = mode * 1000003ull + blockIdx.x * blockDim.x + threadIdx.x;
  rnd(s);
  for (int it = 0; it < 64; ++it) {
    float e[3], delta = 0.0f, beta = 3.0f;
    uint32_t count = 1u + rnd(s) % 2048u;
    const int span = mode == 1 ? 250 : mode == 2 ? 60 : 8, mid = mode == 1 ? 127 : 120;  // binary exponents
    for (int a = 0; a < 3; ++a) {
      const int x = mid - span / 2 + (int)(rnd(s) % (uint32_t)span);
      e[a] = __uint_as_float((uint32_t)(x < 1 ? 1 : x) << 23 | (rnd(s) & 0x7FFFFFu));
    }
    if (mode == 2) {  // flat and linear leaves, any count and beta
      delta = __uint_as_float((60u + rnd(s) % 60u) << 23 | (rnd(s) & 0x7FFFFFu));
      if (rnd(s) & 1u) e[rnd(s) % 3u] = 0.0f;
      count = 1u + (rnd(s) >> (rnd(s) % 31u));
      beta = __uint_as_float((110u + rnd(s) % 30u) << 23 | (rnd(s) & 0x7FFFFFu));
    }
    if (mode == 3) {  // exact cube roots: equal extents, cubic counts
      const uint32_t m = 1u + rnd(s) % 256u;
      count = m * m * m;
      e[1] = e[2] = e[0];
      beta = 1.0f;
    }
    float H[3];
    for (int a = 0; a < 3; ++a) H[a] = e[a] < delta ? delta : e[a];
    const float x = leaf_voxel_size(e, delta, count, beta), y = leaf_voxel_size_fp64(H[0], H[1], H[2], count, beta);
    if (__float_as_uint(x) != __float_as_uint(y)) atomicAdd(bad, 1ull);
  }
}
int main(int, char **v) {
  unsigned long long *bad;
  cudaMallocManaged(&bad, 8);
  *bad = 0;
  k_compare<<<2048, 128>>>(atoi(v[1]), bad);
  if (cudaDeviceSynchronize() != cudaSuccess) return 2;
  printf("%llu\n", *bad);
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_2512_10386_gb300 import build
    d = tmp_path_factory.mktemp("voxel")
    (d / "voxel.cu").write_text(PROGRAM)
    subprocess.run([build._nvcc(), *build.NVCC_FLAGS, str(d / "voxel.cu"), "-o", str(d / "voxel")], check=True)
    return d / "voxel"


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
def test_bits_of_the_definition(program, mode):
    r = subprocess.run([str(program), str(mode)], capture_output=True, text=True, check=True)
    assert int(r.stdout) == 0
