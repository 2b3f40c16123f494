"""The reciprocal square root of the Cholesky pivots (csrc/rsqrt.cuh) over the whole normal range of FP64,
at both ends of every binade and below the range, against 1 / sqrt(x) in extended precision and against
CUDA's own rsqrt. The iteration's remainder is 2^-66; its last step rounds once and adds a term of 2^-22
of the result that carries a few roundings: half a unit in the last place and little more, 0.51. CUDA
states one unit for its function."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "rsqrt.cuh"
__global__ void k(const double* x, double* a, double* b, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    a[i] = fpeps::rsqrt_fast(x[i]);
    b[i] = rsqrt(x[i]);
  }
}
extern "C" int run(const double* x, double* a, double* b, int n) {
  k<<<(n + 255) / 256, 256>>>(x, a, b, n);
  return (int)cudaDeviceSynchronize();
}
"""


def test_rsqrt_over_its_range(tmp_path):
    import torch
    from paper_2511_01039_gb300 import build
    src, so = tmp_path / "r.cu", tmp_path / "r.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc()] + build.flags() + ["-shared", str(src), "-o", str(so)], check=True)
    g = np.random.default_rng(0)
    e = np.repeat(np.arange(-1022, 1024), 500)
    m = 1 + g.random(e.size)
    m[::5] = 1 + g.integers(0, 4, m[::5].size) * 2.0 ** -52       # first numbers of a binade
    m[1::5] = 2 - g.integers(1, 5, m[1::5].size) * 2.0 ** -52     # and last ones
    x = np.concatenate([np.ldexp(m, e), [5e-324, 1e-310, 2.2250738585072009e-308]])
    d = [torch.tensor(x, device="cuda"), *(torch.empty(x.size, dtype=torch.float64, device="cuda") for _ in range(2))]
    fn = ctypes.CDLL(str(so)).run
    assert fn(*(ctypes.c_void_p(t.data_ptr()) for t in d), x.size) == 0
    a, b = d[1].cpu().numpy(), d[2].cpu().numpy()
    ref = 1 / np.sqrt(x.astype(np.longdouble))
    ulp = np.spacing(ref.astype(np.float64)).astype(np.longdouble)
    err = np.abs(a.astype(np.longdouble) - ref) / ulp
    normal = x >= 2.0 ** -1022
    assert err[normal].max() < 0.51
    assert err.max() <= 1 and (np.abs(a - b) <= np.spacing(b)).all()
