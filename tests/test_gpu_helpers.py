"""The reciprocals, roots and exponentials that the kernels build on the hardware's
approximate operations, compiled from their own headers: the FP64 ones against long
double within the error that their one Householder step leaves, the FP32 ones against
CUDA's functions on normal arguments, bit for bit."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SOURCE = r"""
#include "pair_f64.cuh"
using namespace c8r;
template <class F>
__global__ void k_map1(const double* a, double* o, int n, F f) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) o[i] = f(a[i]);
}
__global__ void k_f32(const float* a, const float* b, float* o, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  o[i] = rsqrt_ap(a[i]);
  o[n + i] = rsqrtf(a[i]);
  o[2 * n + i] = div_ap(a[i], b[i]);
  o[3 * n + i] = __fdividef(a[i], b[i]);
  const float x = 80.0f * (2.0f * b[i] / (1.0f + b[i]) - 1.0f);  // b > 0: within +-80
  o[4 * n + i] = exp_ap(x);
  o[5 * n + i] = __expf(x);
}
struct Rsqrt { __device__ double operator()(double x) const { return rsqrt_f64(x); } };
struct Rcp { __device__ double operator()(double x) const { return rcp_f64(x); } };
extern "C" int run_f64(int which, const double* a, double* o, int n) {
  const int blocks = (n + 255) / 256;
  if (which == 0) k_map1<<<blocks, 256>>>(a, o, n, Rsqrt{}); else k_map1<<<blocks, 256>>>(a, o, n, Rcp{});
  return cudaDeviceSynchronize();
}
extern "C" int run_f32(const float* a, const float* b, float* o, int n) {
  k_f32<<<(n + 255) / 256, 256>>>(a, b, o, n);
  return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2309_03717_gb300 import build
    d = tmp_path_factory.mktemp("helpers")
    src, so = str(d / "helpers.cu"), str(d / "helpers.so")
    open(src, "w").write(SOURCE)
    # the FP64 units' flags
    subprocess.run([build.nvcc(), *build.ARCH, *build.COMMON, "--fmad=false", "-I", build.CSRC, "-shared", src, "-o", so],
                   check=True, capture_output=True, text=True, cwd=os.path.dirname(src))
    out = ctypes.CDLL(so)
    P = ctypes.c_void_p
    out.run_f64.argtypes = [ctypes.c_int, P, P, ctypes.c_int]
    out.run_f32.argtypes = [P, P, P, ctypes.c_int]
    return out


@pytest.mark.parametrize("which,low,high", [(0, -1021.0, 1023.0), (0, -40.0, 60.0), (1, -1020.0, 1020.0), (1, -40.0, 40.0)])
def test_fp64_reciprocal_and_root(lib, which, low, high):
    """From y with e = 1 - x y^2 (or 1 - x r) of 2^-20 or less.  Root: 5/16 e^3 is left
    and x y is rounded before it enters e, 2^-53/2 of y, then the sum's half ulp: one
    ulp (and 1 % for the terms of e).  Reciprocal: e is exact but for 2^-73, e^3 is
    left: half an ulp (and 2 %: 2^-60 is 2^-7 of an ulp at most)."""
    rng = np.random.default_rng(which)
    x = np.exp2(rng.uniform(low, high, 1 << 20))
    x[:4096] = np.nextafter(np.exp2(np.round(np.log2(x[:4096]))), rng.choice([0.0, np.inf], 4096))  # around powers of two
    if which == 1:
        x = x * rng.choice([-1.0, 1.0], len(x))
    a = torch.from_numpy(x).cuda()
    o = torch.empty_like(a)
    assert lib.run_f64(which, a.data_ptr(), o.data_ptr(), len(x)) == 0
    X = x.astype(np.longdouble)
    want = 1 / np.sqrt(X) if which == 0 else 1 / X
    err = np.abs((o.cpu().numpy().astype(np.longdouble) - want) / np.spacing(np.abs(want).astype(np.float64)))
    assert float(err.max()) <= (1.01 if which == 0 else 0.52), float(err.max())


def test_fp32_approximations_are_the_cuda_functions(lib):
    n = 1 << 22
    g = torch.Generator(device="cuda").manual_seed(3)
    a, b = (torch.exp2(80.0 * torch.rand(n, generator=g, device="cuda") - 40.0) for _ in range(2))
    o = torch.empty((6, n), device="cuda")
    assert lib.run_f32(a.data_ptr(), b.data_ptr(), o.data_ptr(), n) == 0
    for k, name in ((0, "rsqrt"), (2, "quotient"), (4, "exponential")):
        assert torch.isfinite(o[k]).all() and torch.equal(o[k], o[k + 1]), name
