"""The FP64 reciprocals and reciprocal square roots that the kernels iterate from the hardware's 20-bit seeds, in
their device form, against correctly rounded quotients (numpy) and roots in extended precision.  A reciprocal's last
step is one fused multiply-add on a term exact to 2^-60: half an ulp, and the reference's half.  A reciprocal root's
residual 1 - x y^2 carries the rounding of x y, half an ulp of 1, which counts by half: three quarters of an
ulp, and the reference in extended precision.  So 2^-52 relative in both, for arguments and results over the normal
range; every mantissa pattern class: random, powers of two and their neighbours."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1603_06855_gb300", "csrc")
HARNESS = r"""
#include "mma_update.cuh"
#include "small_dense.cuh"
__global__ void k_math(int what, long long n, const double* x, double* y) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if (what == 0) y[i] = mma_inv(x[i]);
  else if (what == 1) y[i] = inv_newton(x[i]);
  else if (what == 2) y[i] = mma_rsqrt(x[i]);
  else y[i] = inv_sqrt(x[i]);
}
extern "C" int run(int what, long long n, const double* x, double* y) {
  k_math<<<(unsigned)((n + 255) / 256), 256>>>(what, n, x, y);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_06855_gb300 import build_lib
    nvcc = build_lib._nvcc()
    if shutil.which(nvcc) is None:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("device_math")
    src, lib = d / "h.cu", d / "libh.so"
    src.write_text(HARNESS)
    subprocess.run([nvcc, *build_lib.ARCH, *build_lib.FLAGS, "-shared", "-I", CSRC, str(src), "-o", str(lib)], check=True,
                   capture_output=True)
    so = ctypes.CDLL(str(lib))
    so.run.argtypes = [ctypes.c_int, ctypes.c_longlong, ctypes.c_void_p, ctypes.c_void_p]

    def go(what, x):
        t = torch.from_numpy(x).cuda()
        y = torch.empty_like(t)
        torch.cuda.synchronize()
        assert so.run(what, t.numel(), t.data_ptr(), y.data_ptr()) == 0
        return y.cpu().numpy()
    return go


def arguments(e):
    rng = np.random.default_rng(e)
    m = 1.0 + rng.uniform(0, 1, 1 << 19)
    x = np.ldexp(m, rng.integers(-e, e, m.size))
    p = np.ldexp(1.0, np.arange(-e, e))
    near = np.concatenate([np.ldexp(1.0 + np.arange(-64, 65) * 2.0**-52, k) for k in (-e, -1, 0, 1, 2, e - 1)])
    return np.concatenate([x, p, np.nextafter(p, 0), np.nextafter(p, np.inf), near, m])


@pytest.mark.parametrize("what", [0, 1])
def test_reciprocals(run, what):
    x = arguments(1000)
    ref = 1.0 / x
    assert np.all(np.abs(run(what, x) - ref) <= 2.0**-52 * ref)


@pytest.mark.parametrize("what", [2, 3])
def test_reciprocal_roots(run, what):
    x = arguments(1000)
    ref = 1 / np.sqrt(x.astype(np.longdouble))
    assert np.all(np.abs(run(what, x).astype(np.longdouble) - ref) <= 2.0**-52 * ref)
