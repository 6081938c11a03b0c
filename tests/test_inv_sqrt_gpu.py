"""inv_sqrt (csrc/inv_sqrt.cuh) equals the two correctly rounded operations it stands
for, 1.0f / sqrtf(x), bit for bit, on every positive FP32 value, zero and infinity
included: the Cholesky pivots and the Jacobi rotations rest on it."""
import subprocess

import pytest

from paper_2002_08014_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cstdio>
#include "inv_sqrt.cuh"
__global__ void compare(unsigned count, unsigned* bad, unsigned* where) {
  for (unsigned u = blockIdx.x * blockDim.x + threadIdx.x; u < count; u += gridDim.x * blockDim.x) {
    const float x = __uint_as_float(u);
    if (__float_as_uint(lp::inv_sqrt(x)) != __float_as_uint(1.0f / sqrtf(x))) {
      atomicAdd(bad, 1u);
      atomicMin(where, u);
    }
  }
}
int main() {
  unsigned *p, h[2] = {0u, ~0u};
  if (cudaMalloc(&p, 8) || cudaMemcpy(p, h, 8, cudaMemcpyHostToDevice)) return 2;
  compare<<<1024, 256>>>(0x7F800001u, p, p + 1);
  if (cudaMemcpy(h, p, 8, cudaMemcpyDeviceToHost)) return 2;
  printf("%u %08x\n", h[0], h[1]);
  return 0;
}
"""


def test_inv_sqrt_on_every_positive_value(gpu_lib, tmp_path):
    src, exe = tmp_path / "sweep.cu", tmp_path / "sweep"
    src.write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, *build.CFLAGS, str(src), "-o", str(exe)], check=True,
                   capture_output=True, text=True)
    r = subprocess.run([str(exe)], check=True, capture_output=True, text=True)
    assert r.stdout.split() == ["0", "ffffffff"]
