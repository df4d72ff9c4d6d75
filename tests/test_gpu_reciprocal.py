"""reciprocal() of csrc/dgpe_device.cuh (U(k) of the FP32 z pass) over the range of k^2, against exact products."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "dgpe_device.cuh"
static __global__ void k(const float *x, float *r, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) r[i] = dgpe::reciprocal(x[i]);
}
extern "C" int run(const float *x, float *r, int n) {
  k<<<(n + 255) / 256, 256>>>(x, r, n);
  return (int)cudaDeviceSynchronize();
}
"""


def test_reciprocal_is_within_half_an_ulp_of_one(tmp_path):
    import torch
    from paper_1601_04640_gb300 import build as gbuild
    src, lib = str(tmp_path / "reciprocal.cu"), str(tmp_path / "libreciprocal.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([gbuild._nvcc(), *gbuild.ARCH, *gbuild.FLAGS, "-shared", src, "-o", lib], check=True)
    run = ctypes.CDLL(lib).run
    rng = np.random.default_rng(3)
    # k^2 relative to the largest step: from one step along the finest of very uneven axes to 3 256^2, and far beyond
    x = np.concatenate([np.exp2(rng.uniform(-60, 20, 1 << 20)), np.exp2(rng.uniform(-100, 100, 1 << 18)),
                        np.exp2(np.arange(-100.0, 101.0)), np.nextafter(np.float32(2.0), 0) * np.exp2(np.arange(-100.0, 100.0))])
    x = torch.from_numpy(x.astype(np.float32)).cuda()
    r = torch.empty_like(x)
    assert run(ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(r.data_ptr()), x.numel()) == 0
    e = float((x.double() * r.double() - 1.0).abs().max())  # the product is exact in 64 bits
    # a rounding of the result, at most 2^-24 of it; the squared error of the approximation and the rounding of its
    # residual, 2^-44 and 2^-46
    print("max |x r - 1| / 2^-24:", e * 2.0 ** 24)
    assert e <= 2.0 ** -24 + 2.0 ** -44 + 2.0 ** -46
