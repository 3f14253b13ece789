"""The scan's check-free division and square root (div_log, sqrt_bm,
div_range in sg_device.cuh) equal the IEEE operations bit for bit over every
operand they are called with."""

from __future__ import annotations

import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2305_04180_gb300 import build

SRC = r"""
#include <cuda_runtime.h>
#include "sg_device.cuh"
using namespace sg;
__device__ unsigned long long bad[3];
__device__ void cmp(int w, float a, float b) {
  if (__float_as_uint(a) != __float_as_uint(b)) atomicAdd(&bad[w], 1ull);
}
// every mantissa m of f_log's reduction, every 24-bit uniform draw
__global__ void k_unit() {
  const uint32_t b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < (1u << 23)) {
    float m = __uint_as_float(b | 0x3F800000u);
    if (m > 1.41421356237310f) m = m * 0.5f;
    cmp(0, div_log(m - 1.0f, m + 1.0f), __fdiv_rn(m - 1.0f, m + 1.0f));
  }
  const float l = f_log((float)(b + 1u) * kTwoPow24Inv);
  cmp(1, sqrt_bm(-2.0f * l), __fsqrt_rn(-2.0f * l));
}
// every float in [lo, range_max], and zero
__global__ void k_range(uint32_t lo, uint32_t n, float rm, float zh, float zl) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += gridDim.x * blockDim.x) {
    const float r = i == n ? 0.0f : __uint_as_float(lo + i);
    cmp(2, div_range(r, rm, zh, zl), __fdiv_rn(r, rm));
  }
}
extern "C" int run(const float* rm, int n_rm, float lo, unsigned long long* out) {
  k_unit<<<(1 << 24) / 256, 256>>>();
  for (int i = 0; i < n_rm; ++i) {
    const float zh = 1.0f / rm[i], zl = (float)(1.0 / (double)rm[i] - (double)zh);
    union { float f; uint32_t u; } a = {lo * rm[i]}, b = {rm[i]};
    k_range<<<4096, 256>>>(a.u, b.u - a.u + 1u, rm[i], zh, zl);
  }
  cudaError_t e = cudaMemcpyFromSymbol(out, bad, sizeof(bad));
  return (int)e;
}
"""


@pytest.mark.gpu
def test_scan_division_and_square_root_equal_ieee(tmp_path):
    src, lib = tmp_path / "m.cu", tmp_path / "libm.so"
    src.write_text(SRC)
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-fmad=false", "-Xcompiler", "-fPIC",
                    "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC, "-shared", str(src), "-o", str(lib)],
                   check=True)
    rm = np.array([100.0, 99.99999, 1.0, 2.0 ** -20, 3.0e-5, 0.3, 366.7, 4096.0, 12345.678, 2.0 ** 20], np.float32)
    out = np.zeros(3, np.uint64)
    rc = C.CDLL(str(lib)).run(rm.ctypes.data_as(C.c_void_p), C.c_int(rm.size), C.c_float(2.0 ** -24),
                              out.ctypes.data_as(C.c_void_p))
    assert rc == 0
    assert out.tolist() == [0, 0, 0]
