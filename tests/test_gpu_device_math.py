"""Device functions of the kernels (csrc/rgb_kernels.cuh, csrc/misc_kernels.cuh) value by value, from a small library of
their own: the FP64 quotient of the low modes and the FP32 scaling of paths against numpy."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "misc_kernels.cuh"
#include "rgb_kernels.cuh"
using namespace dynot;
__global__ void quot(int n, const double* a, const double* b, double* q) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) q[i] = quot_low(a[i], b[i]);
}
__global__ void scale(int n, const float* v, double s, float sh, float sl, float* o) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) o[i] = scaled<float>(v[i], s, sh, sl);
}
extern "C" int run_quot(int n, const double* a, const double* b, double* q) {
  quot<<<(n + 255) / 256, 256>>>(n, a, b, q);
  return (int)cudaDeviceSynchronize();
}
extern "C" int run_scale(int n, const float* v, double s, float* o) {
  const float sh = (float)s, sl = (float)(s - (double)sh);
  scale<<<(n + 255) / 256, 256>>>(n, v, s, sh, sl, o);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_04840_gb300 import _build
    d = tmp_path_factory.mktemp("math")
    (d / "math.cu").write_text(SRC)
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    subprocess.run([nvcc, *_build.FLAGS, "-shared", "-I", _build.CSRC, "-o", str(d / "math.so"), str(d / "math.cu")],
                   check=True)
    return ctypes.CDLL(str(d / "math.so"))


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def test_low_mode_quotient(lib):
    """Numerators of any sign and size, eigenvalues from 1e-6 to 64 (the largest threshold of the plans): two units in the
    last place of FP64."""
    import torch
    rng = np.random.default_rng(1)
    n = 200000
    a = rng.standard_normal(n) * 10.0 ** rng.uniform(-30, 30, n)
    b = 10.0 ** rng.uniform(-6, np.log10(64.0), n)
    q = torch.empty(n, dtype=torch.float64, device="cuda")
    ta, tb = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    assert lib.run_quot(n, _p(ta), _p(tb), _p(q)) == 0
    assert np.max(np.abs(q.cpu().numpy() / (a / b) - 1)) <= 2.0 ** -51


@pytest.mark.parametrize("s", [1.0, 1.0 / 3.0, 7.31e-6, 12345.678, 3e17])
def test_scaled_path(lib, s):
    """The FP64 product rounded to FP32 once: half a unit in the last place, and the infinities and NaN of that product."""
    import torch
    rng = np.random.default_rng(3)
    v = (rng.standard_normal(100000) * 10.0 ** rng.uniform(-20, 20, 100000)).astype(np.float32)
    v[:8] = [np.inf, -np.inf, np.nan, 3.4e38, -3.4e38, 1e30, 0.0, -0.0]
    tv = torch.from_numpy(v).cuda()
    to = torch.empty_like(tv)
    assert lib.run_scale(len(v), _p(tv), ctypes.c_double(s), _p(to)) == 0
    o = to.cpu().numpy()
    exact = v.astype(np.float64) * s
    with np.errstate(over="ignore"):
        want = exact.astype(np.float32)
    fine = np.isfinite(want)
    assert np.array_equal(o[~fine], want[~fine], equal_nan=True)
    ulp = np.spacing(np.abs(want[fine]).astype(np.float32)).astype(np.float64)
    assert np.all(np.abs(o[fine].astype(np.float64) - exact[fine]) <= 0.5000001 * ulp)
