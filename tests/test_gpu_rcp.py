"""The FP64 reciprocal of the Cholesky panels (csrc/rcp.cuh) over its whole range, against exact
quotients. Compiled here into a small library around the header.

Bound, derived before the first run: the seed is within 2^-21, so e^3 < 2^-63 is left before the
last rounding, and the rounding of the correction r (e + e^2) is below 2^-53 2^-20 of r: the
relative error is at most 2^-53 (1 + 2^-8)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

SOURCE = r"""
#include <cuda_runtime.h>
#include "rcp.cuh"
__global__ void apply(const double *x, double *y, int *in, int n) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  in[i] = hatt::rcp_range(x[i]);
  y[i] = in[i] ? hatt::rcp_seeded(x[i]) : 0.0;
}
extern "C" int rcp(const double *x, double *y, int *in, int n) {
  apply<<<(n + 255) / 256, 256>>>(x, y, in, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def rcp(tmp_path_factory):
    from paper_2410_04385_gb300 import build
    d = tmp_path_factory.mktemp("rcp")
    src, lib = str(d / "rcp.cu"), str(d / "librcp.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build.nvcc_path(), build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                    "-I" + build.CSRC, src, "-o", lib], check=True)
    fn = ctypes.CDLL(lib).rcp

    def call(x):
        xd = torch.from_numpy(x).cuda()
        y, inside = torch.zeros_like(xd), torch.zeros(len(x), dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert fn(ctypes.c_void_p(xd.data_ptr()), ctypes.c_void_p(y.data_ptr()),
                  ctypes.c_void_p(inside.data_ptr()), len(x)) == 0
        return y.cpu().numpy(), inside.cpu().numpy().astype(bool)

    return call


def error(x, y):
    """|x y - 1| from the products' exact halves (x y is within a few roundings of 1)."""
    def halves(v):
        hi = (v.view(np.uint64) & np.uint64(0xFFFFFFFFF8000000)).view(np.float64)
        return hi, v - hi
    (a, b), (c, d) = halves(x), halves(y)
    return np.abs(((a * c - 1.0) + a * d + b * c) + b * d)


def test_reciprocal_over_its_range(rcp):
    rng = np.random.default_rng(1)
    p = 2.0 ** np.arange(-100, 100)
    edge = np.concatenate([p, np.nextafter(p, 2 * p), np.nextafter(2 * p, p), p * 1.5,
                           np.nextafter(p * 1.5, p), p * (2 - 2.0 ** -22), p * (1 + 2.0 ** -23), p * (1 + 2.0 ** -24)])
    x = np.concatenate([edge, rng.uniform(1, 2, 1 << 20) * 2.0 ** rng.integers(-100, 100, 1 << 20)])
    y, inside = rcp(x)
    assert inside.all()
    assert np.all(error(x, y) <= 2.0 ** -53 * (1 + 2.0 ** -8))


def test_values_outside_are_told_apart(rcp):
    x = np.array([0.0, -0.0, -1.0, -2.0 ** -80, 2.0 ** 100, np.nextafter(2.0 ** -100, 0), 5e-324, 1e-300, 1e300,
                  np.inf, -np.inf, np.nan])
    assert not rcp(x)[1].any()
