"""The reflectors' roots and inverses (csrc/roots.cuh) against correctly rounded ones, over every binary exponent
of float and double, subnormal numbers and infinity included."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from tests.gpu_common import cuda_or_skip

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "roots.cuh"
__device__ float seed(float x) { return rsqrtf(x); }
__device__ double seed(double x) { return rsqrt(x); }
__device__ float seed_ftz(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ float rcp(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ double rcp(double x) { return 1.0 / x; }
template <typename T>
__global__ void roots(const T* x, T* out, long long n) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  T y = seed(x[i]);
  if (sizeof(T) == 4 && x[i] >= T(1.17549435e-38)) y = seed_ftz(x[i]);
  const T r = qrkit::dev::newton_root(x[i], y);
  out[i] = r;
  out[n + i] = qrkit::dev::newton_inverse(r, y);
  out[2 * n + i] = qrkit::dev::newton_inverse(r, rcp(r));
}
extern "C" int run(int dbl, const void* x, void* out, long long n) {
  if (dbl) roots<double><<<(unsigned)((n + 255) / 256), 256>>>((const double*)x, (double*)out, n);
  else roots<float><<<(unsigned)((n + 255) / 256), 256>>>((const float*)x, (float*)out, n);
  return (int)cudaDeviceSynchronize();
}
"""


# a seed within 2^-21 leaves an error of 2^-41 after the step, so the rounding of the last operation decides: the root
# within one unit in the last place.  The inverse is that of the rounded root (half a unit) and rounded once: two units
# of the inverse of the exact root
@pytest.mark.parametrize("dtype,lo,hi", [(np.float32, -149, 128), (np.float64, -1074, 1024)])
def test_roots_within_an_ulp(tmp_path, dtype, lo, hi):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import build
    (tmp_path / "roots.cu").write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-I", build.CSRC, "-shared", "-Xcompiler", "-fPIC",
                    "-o", str(tmp_path / "roots.so"), str(tmp_path / "roots.cu")], check=True, capture_output=True)
    fn = ctypes.CDLL(os.path.join(tmp_path, "roots.so")).run
    fn.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong]
    g = np.random.default_rng(0)
    e = np.repeat(np.arange(lo, hi), 3000)
    m = 1.0 + g.random(e.size)
    m[::3000], m[1::3000] = 1.0, np.nextafter(dtype(2), dtype(1))
    with np.errstate(under="ignore"):
        x = np.ldexp(m.astype(dtype), e).astype(dtype)
    x = x[(x > 0) & np.isfinite(x)]
    xs = torch.from_numpy(np.concatenate([x, [np.inf]]).astype(dtype)).cuda()
    out = torch.empty(3, xs.numel(), dtype=xs.dtype, device="cuda")
    assert fn(int(dtype is np.float64), xs.data_ptr(), out.data_ptr(), xs.numel()) == 0
    r, inv, inv2 = out.cpu().numpy()
    assert np.isinf(r[-1]) and inv[-1] == 0
    exact = np.sqrt(x.astype(np.longdouble))
    ulp = np.spacing(exact.astype(dtype)).astype(np.longdouble)
    assert (np.abs(r[:-1] - exact) / ulp).max() <= 1.0
    iulp = np.spacing((1 / exact).astype(dtype)).astype(np.longdouble)
    for v in (inv, inv2):
        assert (np.abs(v[:-1] - 1 / exact) / iulp).max() <= 2.0
