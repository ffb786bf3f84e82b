"""The refined reciprocal and inverse square root of site.cuh by themselves (GPU).

FP64: one step of third order from the hardware's approximation.  The last
multiply-add rounds once (2^-53), the residual of 1 / sqrt(a) carries the
rounding of a y (another 2^-54 of the result), and the third-order remainder is
below 2^-54: 2^-52 in all.  FP32: the hardware's 1 ulp and rsqrtf's 2 ulp.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "site.cuh"
template <typename T> __global__ void k_both(const T* a, T* r, T* s, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  r[i] = rlbm::qrcp(a[i]);
  s[i] = rlbm::qrsqrt(a[i]);
}
extern "C" int both64(const double* a, double* r, double* s, int n) {
  k_both<double><<<(n + 127) / 128, 128>>>(a, r, s, n);
  return (int)cudaDeviceSynchronize();
}
extern "C" int both32(const float* a, float* r, float* s, int n) {
  k_both<float><<<(n + 127) / 128, 128>>>(a, r, s, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_02418_gb300 import build
    d = tmp_path_factory.mktemp("recip")
    src, out = str(d / "recip.cu"), str(d / "librecip.so")
    open(src, "w").write(SOURCE)
    subprocess.run([build.nvcc(), "-shared", "-O3", "-std=c++17", "-I" + build.CSRC, *build.ARCH, "-fmad=false",
                    "-Xcompiler", "-fPIC", "-o", out, src], check=True, capture_output=True)
    return torch, ctypes.CDLL(out)


def run(lib, name, a):
    torch, so = lib
    x = torch.tensor(a, device="cuda")
    r, s = torch.empty_like(x), torch.empty_like(x)
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    torch.cuda.synchronize()
    assert getattr(so, name)(p(x), p(r), p(s), x.numel()) == 0
    return r.cpu().numpy(), s.cpu().numpy()


@pytest.mark.parametrize("name,dtype,exps,bound_r,bound_s", [
    ("both64", np.float64, (-1000, 1000), 2.0 ** -52, 2.0 ** -52),
    ("both32", np.float32, (-120, 120), 2.0 ** -23, 2.0 ** -22)])
def test_relative_errors(lib, name, dtype, exps, bound_r, bound_s):
    rng = np.random.default_rng(0)
    n = 200_000
    a = np.concatenate([
        rng.uniform(1, 4, n),                                          # one binade pair, densely
        np.ldexp(rng.uniform(1, 2, n), rng.integers(*exps, n)),        # the whole range
        1 + np.linspace(-1e-3, 1e-3, n),                               # near rest
        np.ldexp(1.0, np.arange(*exps)),                               # powers of two
        1 - np.ldexp(rng.uniform(0.5, 1, n), rng.integers(-24, 0, n)),   # 1 - u^2
    ]).astype(dtype)
    a = a[a > 0]
    r, s = run(lib, name, a)
    w = a.astype(np.longdouble)        # at least 64 bits of mantissa
    err_r = np.abs(r.astype(np.longdouble) * w - 1)
    err_s = np.abs(s.astype(np.longdouble) * np.sqrt(w) - 1)
    slack = 2.0 ** -60 if dtype == np.float64 else 0.0    # roundings of the check itself
    assert float(err_r.max()) <= bound_r + slack
    assert float(err_s.max()) <= bound_s + slack
