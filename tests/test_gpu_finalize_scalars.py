"""The double-precision reciprocal behind the scale of the scores' diversity term,
alone: over the exponents of a double, at random mantissas and next to powers of
two, within 2^-46 of 1 / b (a Newton-Raphson step squares the seed's error, at most
2^-23.4 after the mantissa's rounding to single precision and the reciprocal's)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2609_06663_gb300.build import ARCH, FLAGS, nvcc

pytestmark = pytest.mark.gpu

SOURCE = """
#include "finalize_cluster.cuh"
__global__ void rcp(const double* b, double* r, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) r[i] = ecokv::rcp_double(b[i]);
}
extern "C" int run(const double* b, double* r, int n) {
  rcp<<<(n + 255) / 256, 256>>>(b, r, n);
  return (int)cudaDeviceSynchronize();
}
"""


def test_rcp_double(tmp_path):
    src, so = tmp_path / "rcp.cu", tmp_path / "rcp.so"
    src.write_text(SOURCE)
    subprocess.run([nvcc(), *ARCH, *FLAGS, "-shared", "-cudart", "shared", "-o", os.fspath(so), os.fspath(src)],
                   check=True, capture_output=True, timeout=300)
    g = np.random.default_rng(1)
    b = np.ldexp(1.0 + g.random(1 << 20), g.integers(-1000, 1000, 1 << 20))
    near = np.ldexp(1.0, np.arange(-1000, 1000))
    b = np.concatenate([b, near, np.nextafter(near, np.inf), np.nextafter(near, 0.0)])
    b_dev = torch.from_numpy(b).cuda()
    r_dev = torch.zeros_like(b_dev)
    torch.cuda.synchronize()
    assert ctypes.CDLL(os.fspath(so)).run(ctypes.c_void_p(b_dev.data_ptr()), ctypes.c_void_p(r_dev.data_ptr()),
                                          ctypes.c_int(b.size)) == 0
    r = r_dev.cpu().numpy()
    # 1 / b correctly rounded is itself within 2^-53
    err = np.abs(r / (1.0 / b) - 1.0).max()
    assert err <= 2.0 ** -46, err
