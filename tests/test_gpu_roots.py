"""root_and_inverse (csrc/expand64.cuh), the distance and its reciprocal from the FP32 estimate and
one third-order (Householder) step, against the correctly rounded square root and against 1 / sqrt in
extended precision: over all exponents of r^2 that the FP32 estimate covers and beyond, mantissas at
the ends of a binade and at random.

Bar: the estimate is off by at most 2^-22 (CUDA's bound for rsqrtf: 2 ulp, 2^-23 each, and r^2's
rounding, 2^-25 of the root), so e = 1 - r^2 y^2 is below 2^-20.8 and the series' next term,
5 e^3 / 16, below 2^-64. The product t = r^2 y carries half an ulp, half of which the step takes out;
the last operation rounds once more: 1.5 units of 2^-53 in either result, 1.6 with what is left."""
import ctypes
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SOURCE = """
#include "expand64.cuh"
__global__ void roots(const double* r2, double* r, double* ri, int n) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) bem::root_and_inverse(r2[t], r[t], ri[t]);
}
extern "C" int run(const double* r2, double* r, double* ri, int n) {
  roots<<<(n + 255) / 256, 256>>>(r2, r, ri, n);
  return (int)cudaDeviceSynchronize();
}
"""


def test_against_exact_roots(tmp_path):
    from paper_1906_03938_gb300 import build
    src, lib = tmp_path / "roots.cu", tmp_path / "libroots.so"
    src.write_text(SOURCE)
    subprocess.run([build.NVCC, *build.ARCH, *build.FLAGS, "-shared", str(src), "-o", str(lib)], check=True)
    rs = np.random.RandomState(1)
    e = np.arange(-600, 601)
    m = np.concatenate([1.0 + rs.rand(e.size, 300), np.full((e.size, 1), 1.0),
                        np.full((e.size, 1), 2.0 - 2.0 ** -52), 1.0 + 2.0 ** -np.arange(1, 53) * np.ones((e.size, 1))], 1)
    x = np.ldexp(m, e[:, None]).reshape(-1)
    dx = torch.from_numpy(x).to("cuda:0")
    r, ri = torch.empty_like(dx), torch.empty_like(dx)
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    torch.cuda.synchronize()
    assert ctypes.CDLL(str(lib)).run(p(dx), p(r), p(ri), x.size) == 0
    root = np.sqrt(x.astype(np.longdouble))
    for got, ref in ((r, root), (ri, 1 / root)):
        err = np.abs(got.cpu().numpy().astype(np.longdouble) / ref - 1)
        assert float(err.max()) <= 1.6 * 2.0 ** -53
