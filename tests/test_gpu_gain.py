"""The factor h / (1 + h) of the implicit solve in the complex64 default steps: the division's value for
every finite FP32 h, and steps at an h whose 1 + h is beyond an approximate reciprocal's range."""
import os
import subprocess

import numpy as np
import pytest

import kd_inputs as I

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

EVERY_H = r"""
#include <cstdio>
#include "kd_stage.cuh"
__global__ void compare(unsigned long long* differ) {
  for (unsigned long long i = blockIdx.x * 256ull + threadIdx.x; i < 0x7f800000ull; i += gridDim.x * 256ull) {
    const float h = __uint_as_float((unsigned)i), a = kd::fused_gain(h), b = kd::implicit_gain(h);
    if (__float_as_uint(a) != __float_as_uint(b)) atomicAdd(differ, 1ull);
  }
}
int main() {
  unsigned long long *d = nullptr, n = ~0ull;
  if (cudaMalloc(&d, 8) != cudaSuccess || cudaMemset(d, 0, 8) != cudaSuccess) return 1;
  compare<<<1024, 256>>>(d);
  if (cudaMemcpy(&n, d, 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
  printf("%llu\n", n);
  return 0;
}
"""


def test_gain_is_the_division_for_every_h(tmp_path):
    from paper_1902_00387_gb300 import build as B
    src, exe = tmp_path / "gain.cu", tmp_path / "gain"
    src.write_text(EVERY_H)
    subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-I", B.CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.strip() == "0"


# the persistent step, the 3n/4-point kernels
@pytest.mark.parametrize("n,batch", [(16, 2), (512, 4)])
def test_stiffest_modes_vanish(n, batch):
    """Diffusion alone with dt lambda / 2 from ~1e36 up to 1.1e38 at the highest mode (1 + h passes
    2^126 at three quarters of it, and 1.5 dt lambda stays a finite FP32): a step leaves 1 / (1 + h)^2 of a
    mode or less, zero in FP32."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1902_00387_gb300 as kd
    K, dt = n // 3, 1e3
    Rm = 0.5 * dt * (2 * K * K + 0.57 ** 2) / 1.1e38
    b = torch.tensor(np.stack([I.flat_field(n, 0.57, i) for i in range(batch)]), dtype=torch.complex64, device="cuda")
    y = torch.full_like(b, float("nan"))
    ctx = kd.kd_create(kd.make_params(2, n, 0.57, Rm, dt, kd.KD_C64))
    try:
        kd.kd_fine_batched(ctx, b, y, torch.zeros(batch, dtype=torch.float64, device="cuda"), 1, batch)
        torch.cuda.synchronize()
    finally:
        kd.kd_destroy(ctx)
    assert torch.equal(y, torch.zeros_like(y))
