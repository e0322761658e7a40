"""rsqrt_chain (csrc/common.cuh) against CUDA's correctly rounded __frsqrt_rn: every one of the 2^24
significands of [1, 4), at every power of 4 from 2^-100 to 2^100, bit for bit."""
import ctypes
import subprocess

import pytest

pytestmark = pytest.mark.gpu

COMPARE = r"""
#include "common.cuh"
__global__ void compare(int e4, unsigned long long* differ) {
  const unsigned u = blockIdx.x * 256u + threadIdx.x;  // 0 .. 2^24 - 1: the floats of [1, 4)
  const float v = __uint_as_float(0x3f800000u + u + (unsigned(2 * e4) << 23));
  if (__float_as_uint(dk::rsqrt_chain(v)) != __float_as_uint(__frsqrt_rn(v))) atomicAdd(differ, 1ull);
}
extern "C" __attribute__((visibility("default"))) long long compare_all(int lo4, int hi4) {
  unsigned long long *d, h = ~0ull;
  if (cudaMalloc(&d, sizeof h) != cudaSuccess || cudaMemset(d, 0, sizeof h) != cudaSuccess) return -1;
  for (int e = lo4; e <= hi4; ++e) compare<<<1 << 16, 256>>>(e, d);
  const cudaError_t s = cudaMemcpy(&h, d, sizeof h, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return s == cudaSuccess ? (long long)h : -1;
}
"""


def test_all_significands(tmp_path):
    import torch
    from paper_2602_01330_gb300 import build
    torch.cuda.init()
    src, so = tmp_path / "compare.cu", str(tmp_path / "compare.so")
    src.write_text(COMPARE)
    subprocess.run([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-I", build.CSRC, "-shared", "-cudart", "static",
                    "-o", so, str(src)], check=True, capture_output=True)
    lib = ctypes.CDLL(so)
    lib.compare_all.restype = ctypes.c_longlong
    assert lib.compare_all(-50, 49) == 0  # [2^-100, 2^100)
