"""GELU and GELU' of the GEMM epilogues (gelu2 and gelu_both2 of common.cuh) against the exact functions in
64 bits, in 32 bits as the epilogues hold them (they store bf16): a few lines around the header, compiled
with the library's flags.

Bounds: the absolute errors that the formula which they replace shows on the same grid (Abramowitz & Stegun
7.1.28, the one that ra_eval_activation evaluates), so that no precision is lost by the change."""
import ctypes
import subprocess

import numpy as np
import pytest
from scipy.special import erfc

from paper_2502_19864_gb300 import build as B
from paper_2502_19864_gb300 import ringada as R

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "common.cuh"
__global__ void k(const float2* x, float2* y, float2* y2, float2* d, long n) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  y[i] = ra::gelu2(x[i]);
  ra::gelu_both2(x[i], y2[i], d[i]);
}
extern "C" int run(void* x, void* y, void* y2, void* d, long pairs) {
  k<<<(unsigned)((pairs + 255) / 256), 256>>>((float2*)x, (float2*)y, (float2*)y2, (float2*)d, pairs);
  return (int)cudaDeviceSynchronize();
}
"""


def test_no_further_off_than_the_general_form(tmp_path):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    src, lib = tmp_path / "gelu.cu", tmp_path / "gelu.so"
    src.write_text(SOURCE)
    subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-shared", "-o", str(lib), str(src)], check=True)
    x = torch.linspace(-12, 12, 480000, dtype=torch.float64).float().cuda()
    y, y2, d, y0, d0 = (torch.full_like(x, float("nan")) for _ in range(5))
    run = ctypes.CDLL(str(lib)).run
    assert run(*(ctypes.c_void_p(t.data_ptr()) for t in (x, y, y2, d)), ctypes.c_long(x.numel() // 2)) == 0
    R.ra_eval_activation(0, x.data_ptr(), y0.data_ptr(), x.numel())
    R.ra_eval_activation(1, x.data_ptr(), d0.data_ptr(), x.numel())
    torch.cuda.synchronize()
    v = x.cpu().numpy().astype(np.float64)
    cdf = 0.5 * erfc(-v / np.sqrt(2))
    gelu, grad = v * cdf, cdf + v * np.exp(-v * v / 2) / np.sqrt(2 * np.pi)
    assert torch.equal(y, y2)
    for got, general, ref in ((y, y0, gelu), (d, d0, grad)):
        err, was = (np.abs(t.cpu().numpy().astype(np.float64) - ref) for t in (got, general))
        print("largest %.3g (general form %.3g), rms %.3g (%.3g)" % (
            err.max(), was.max(), np.sqrt((err ** 2).mean()), np.sqrt((was ** 2).mean())))
        assert err.max() <= was.max() and (err ** 2).mean() <= (was ** 2).mean()
