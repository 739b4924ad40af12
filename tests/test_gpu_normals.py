"""The radius of the serial LinGauss actor's Box-Muller pairs is a square root taken by one step of Newton's iteration from the hardware's
reciprocal root (csrc/tj_tc.cuh, normal_radius).  It depends on 23 bits, so every one of its values is compared with sqrtf."""
import ctypes as C
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "tj_tc.cuh"
using namespace tj;
__global__ void radii(unsigned long long* differ) {
  const uint32_t word = (blockIdx.x * blockDim.x + threadIdx.x) << 9;
  float l;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(__uint_as_float((word >> 9) | 0x3F800000u) - 0.99999994f));
  if (normal_radius(word) != sqrtf(l * -1.38629436111989061883f)) atomicAdd(differ, 1ull);
}
extern "C" int run(void* differ) {
  radii<<<(1 << 23) / 256, 256>>>(static_cast<unsigned long long*>(differ));
  return (int)cudaDeviceSynchronize();
}
"""


def test_every_radius_is_correctly_rounded(tmp_path):
    import torch
    from paper_2502_20190_b200 import build
    src, lib = tmp_path / "normals.cu", tmp_path / "normals.so"
    src.write_text(SOURCE)
    subprocess.check_call([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")] + build.NVCC_FLAGS + ["-shared", "-I", build.CSRC, str(src), "-o", str(lib)])
    differ = torch.zeros(1, dtype=torch.int64, device="cuda")
    run = C.CDLL(str(lib)).run
    run.argtypes = [C.c_void_p]
    assert run(differ.data_ptr()) == 0
    assert differ.item() == 0
