"""The FP64 reciprocal and square roots of the pair loops (rcp64, rsqrt64 in
k_pair.cuh) against extended precision on the host, over the squared
distances that a pair can have and far beyond (1e-12 to 1e12).  Derived
bound: the hardware approximation is good to at least 18 bits, the series
step leaves e^3 < 2^-54 of it and one final rounding (half an ulp), the
square root one more in x y: within 1 ulp each."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "k_pair.cuh"
__global__ void k(const double *x, double *o, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double a, b;
  mdk::pair::rsqrt64(x[i], a, b);
  o[i] = mdk::pair::rcp64(x[i]);
  o[n + i] = a;
  o[2 * n + i] = b;
  o[3 * n + i] = mdk::pair::G<mdk::Fp64>::sqr(x[i]);
}
extern "C" int run(const double *x, double *o, int n) {
  k<<<(n + 255) / 256, 256>>>(x, o, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def fn(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_22951_gb300 import _build
    d = tmp_path_factory.mktemp("math")
    src, lib = os.path.join(d, "m.cu"), os.path.join(d, "m.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.NVCC_FLAGS, "-shared", "-I", _build.CSRC,
                    "-I", _build.INCLUDE, src, "-o", lib], check=True, capture_output=True)

    def call(x):
        xd = torch.tensor(x, dtype=torch.float64, device="cuda")
        out = torch.empty(4 * x.size, dtype=torch.float64, device="cuda")
        P = ctypes.c_void_p
        assert ctypes.CDLL(lib).run(P(xd.data_ptr()), P(out.data_ptr()), x.size) == 0
        return out.cpu().numpy().reshape(4, -1)
    return call


def ulps(got, ref):
    return np.max(np.abs(got.astype(np.longdouble) - ref) / np.spacing(np.abs(ref).astype(np.float64)))


@pytest.mark.parametrize("lo,hi", [(1.0, 150.0), (1e-12, 1e12)])
def test_within_one_ulp(fn, lo, hi):
    rng = np.random.default_rng(1)
    x = np.exp(rng.uniform(np.log(lo), np.log(hi), 1 << 20))
    xl = x.astype(np.longdouble)
    rcp, rsq, root, sqr = fn(x)
    assert ulps(rcp, 1 / xl) <= 1.0
    assert ulps(rsq, 1 / np.sqrt(xl)) <= 1.0
    assert ulps(root, np.sqrt(xl)) <= 1.0
    assert np.array_equal(root, sqr)


def test_zero_and_nan(fn):
    rcp, rsq, root, sqr = fn(np.array([0.0, np.nan, np.inf]))
    assert not np.isfinite(rcp[0]) and not np.isfinite(rsq[0])
    assert sqr[0] == 0.0
    assert np.isnan(rcp[1]) and np.isnan(rsq[1]) and np.isnan(sqr[1])
