"""Norms of two floats in double (csrc/roots.cuh), which damp the points' columns of LM steps: over every pair of
magnitudes that floats have, zero and subnormal ones included."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from tests.gpu_common import cuda_or_skip

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "roots.cuh"
__global__ void norms(const float* x, const float* y, double* out, long long n) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) out[i] = qrkit::dev::norm_of_two(x[i], y[i]);
}
extern "C" int run(const float* x, const float* y, double* out, long long n) {
  norms<<<(unsigned)((n + 255) / 256), 256>>>(x, y, out, n);
  return (int)cudaDeviceSynchronize();
}
"""


# two roundings in double (of the sum and of the root, or of the sum of floats that stands for it): within 2^-52
def test_norm_of_two(tmp_path):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import build
    (tmp_path / "norms.cu").write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-I", build.CSRC, "-I",
                    os.path.join(build.ROOT, "include"), "--expt-relaxed-constexpr", "-shared", "-Xcompiler", "-fPIC",
                    "-o", str(tmp_path / "norms.so"), str(tmp_path / "norms.cu")], check=True, capture_output=True)
    fn = ctypes.CDLL(os.path.join(tmp_path, "norms.so")).run
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong]
    g = np.random.default_rng(0)
    n = 400_000
    e = g.integers(-149, 128, size=(2, n))
    e[1, n // 2:] = np.clip(e[0, n // 2:] + g.integers(-30, 31, size=n // 2), -149, 127)   # squares that meet
    with np.errstate(under="ignore"):
        x, y = np.ldexp((1.0 + g.random((2, n))) * g.choice([-1.0, 1.0], (2, n)), e).astype(np.float32)
    x[:1000] = 0.0
    y[500:2000] = 0.0
    tx, ty, out = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), torch.empty(n, device="cuda", dtype=torch.float64)
    torch.cuda.synchronize()
    assert fn(tx.data_ptr(), ty.data_ptr(), out.data_ptr(), n) == 0
    got = out.cpu().numpy()
    want = np.sqrt(x.astype(np.longdouble) ** 2 + y.astype(np.longdouble) ** 2)
    assert (got[want == 0] == 0).all()
    ok = want > 0
    assert (np.abs(got[ok] - want[ok]) / want[ok]).max() <= 2.0 ** -52
