"""The adjoint histograms' fixed-point add (Fx64 in k_adjoint.cu): a float is
rounded to the nearest 64-bit integer, ties to even, exactly -- in the short
form below 2^53, also where the rest beside the high word is a tie of +-2^31,
and in the wide form up to 2^62 -- and sums wrap like integers.  The reference
is exact integer arithmetic on the host."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "k_adjoint.cu"
__global__ void k(const float *x, long long *o, int n, int wide) {
  __shared__ unsigned lo[256];
  __shared__ int hi[256];
  const int t = threadIdx.x;
  const int i = blockIdx.x * 256 + t;
  lo[t] = 0u;
  hi[t] = 0;
  const mdk::Fx64 h{lo, hi};
  if (i >= n) return;
  wide ? h.add<true>(t, x[i]) : h.add<false>(t, x[i]);
  o[i] = h.get(t);
  wide ? h.add<true>(t, -0.75f * x[i]) : h.add<false>(t, -0.75f * x[i]);
  o[n + i] = h.get(t);
}
extern "C" int run(const float *x, long long *o, int n, int wide) {
  k<<<(n + 255) / 256, 256>>>(x, o, n, wide);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def fn(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_22951_gb300 import _build
    d = tmp_path_factory.mktemp("fx")
    src, so = os.path.join(d, "fx.cu"), os.path.join(d, "fx.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.NVCC_FLAGS, "-I", _build.CSRC, "-I",
                    _build.INCLUDE, "-shared", "-o", so, src], check=True)
    torch.zeros(1, device="cuda")
    return ctypes.CDLL(so).run


def nearest(v):
    return round(Fraction(float(v)))         # to even


@pytest.mark.parametrize("wide,top", [(0, 52.9), (1, 62.0)])
def test_rounds_like_an_integer(fn, wide, top):
    import torch
    rng = np.random.default_rng(3)
    x = np.exp2(rng.uniform(-3, top, 4000)) * rng.choice([-1.0, 1.0], 4000)
    k = np.arange(-40, 41) + 0.5             # ties of the high word, rest +-2^31
    halves = np.arange(-40, 41) + 0.5        # ties of the low word
    x = np.concatenate([x, k * 2.0 ** 32, halves, np.arange(-3, 4) * 2.0 ** 31,
                        (2.0 ** 32 + 2.0 ** 31) * np.exp2(np.arange(0, 10))]).astype(np.float32)
    xd = torch.tensor(x, device="cuda")
    out = torch.zeros(2 * len(x), dtype=torch.int64, device="cuda")
    P = ctypes.c_void_p
    assert fn(P(xd.data_ptr()), P(out.data_ptr()), len(x), wide) == 0
    out = out.cpu().numpy().reshape(2, -1)
    for i, v in enumerate(x):
        a = nearest(v)
        assert out[0, i] == a, v
        assert out[1, i] == a + nearest(np.float32(-0.75) * v), v
