"""The flush-to-zero reciprocal square root of the float32 potentials (rsd::inv_sqrt<true>) against rsqrtf,
bit for bit, for every normal positive float32, infinity included: the certified bounds are derived for
either, and the exact list's flags take one member's own term out of sums made with the other."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "rs_common.cuh"
__global__ void k_compare(uint32_t first, uint32_t count, unsigned long long* different) {
  unsigned long long d = 0;
  for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < count; k += gridDim.x * blockDim.x) {
    const float x = __uint_as_float(first + k);
    d += __float_as_uint(rsd::inv_sqrt<true>(x)) != __float_as_uint(rsqrtf(x));
  }
  if (d) atomicAdd(different, d);
}
extern "C" long long compare(uint32_t first, uint32_t count) {
  unsigned long long* d = nullptr;
  unsigned long long h = ~0ull;
  if (cudaMalloc(&d, 8) != cudaSuccess) return -1;
  cudaMemset(d, 0, 8);
  k_compare<<<1216, 256>>>(first, count, d);
  const bool ok = cudaGetLastError() == cudaSuccess && cudaMemcpy(&h, d, 8, cudaMemcpyDeviceToHost) == cudaSuccess;
  cudaFree(d);
  return ok ? (long long)h : -1;
}
"""


def test_flush_to_zero_form_has_the_same_values(tmp_path):
    from paper_2412_18629_gb300 import build
    src, lib = tmp_path / "rsqrt.cu", tmp_path / "rsqrt.so"
    src.write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, *build.NVFLAGS, "-I", build.CSRC, "-shared", "-o", str(lib), str(src)],
                   check=True, cwd=os.path.dirname(build.CSRC))
    compare = ctypes.CDLL(str(lib)).compare
    compare.restype, compare.argtypes = ctypes.c_longlong, [ctypes.c_uint32, ctypes.c_uint32]
    least, inf = 0x00800000, 0x7F800000  # the smallest normal value, infinity
    assert compare(least, inf - least + 1) == 0
