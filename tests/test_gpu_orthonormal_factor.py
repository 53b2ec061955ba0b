"""The factor with which the FP64 projected problems make the FP32 stage's eigenvectors orthonormal: where it is accepted,
the columns are orthonormal to FP64's rounding; where the columns are too far off for its series, it is refused
(the problem is then diagonalised in FP64 from the start).  Columns off by 1e-7 to 5e-4, by an infinity and a NaN.
What a product of n terms rounds to here is below sqrt(n) 2.2e-16 a few times over, and 1e-15 of the series may be
left: 5e-15.  The FP32 stage leaves up to 3.4e-6 at n = 72, in entries of random sign and mostly far smaller (row sums of
E^2 of 2e-11): a tenth of that largest entry throughout must be accepted."""
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
#include "jacobi.cuh"
constexpr int T = 256;
__global__ __launch_bounds__(T) void k_factor(int n, const double2* X, float2* F, double2* E, double2* Q, int* ok) {
  for (int t = threadIdx.x; t < n * n; t += T) {
    const int i = t / n, j = t % n;
    double2 g = make_double2(i == j ? -1.0 : 0.0, 0.0);
    for (int p = 0; p < n; ++p) cfmac(g, X[p * n + i], X[p * n + j]);
    E[t] = g;
    F[i * SR_LD + j] = make_float2((float)g.x, (float)g.y);
  }
  __syncthreads();
  const bool good = orthonormal_factor<T>(F, E, n, n);
  if (threadIdx.x == 0) *ok = good;
  for (int t = threadIdx.x; t < n * n; t += T) {
    double2 g = make_double2(0.0, 0.0);
    for (int p = 0; p < n; ++p) cfma(g, X[t / n * n + p], E[p * n + t % n]);
    Q[t] = g;
  }
}
extern "C" int run(int n, const void* X, void* F, void* E, void* Q, int* ok) {
  k_factor<<<1, T>>>(n, (const double2*)X, (float2*)F, (double2*)E, (double2*)Q, ok);
  return (int)cudaDeviceSynchronize();
}
extern "C" int stride() { return SR_LD; }
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_06855_gb300 import build_lib
    nvcc = build_lib._nvcc()
    if shutil.which(nvcc) is None:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("factor")
    src, lib = d / "h.cu", d / "libh.so"
    src.write_text(HARNESS)
    subprocess.run([nvcc, *build_lib.ARCH, *build_lib.FLAGS, "-shared", "-I", CSRC, str(src), "-o", str(lib)], check=True,
                   capture_output=True)
    so = ctypes.CDLL(str(lib))

    def go(X):
        n = X.shape[0]
        x = torch.from_numpy(np.ascontiguousarray(X)).cuda()
        F = torch.zeros(n * so.stride() * 2, dtype=torch.float32, device="cuda")
        E, Q = torch.empty_like(x), torch.empty_like(x)
        ok = torch.empty(1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert so.run(n, *[ctypes.c_void_p(t.data_ptr()) for t in (x, F, E, Q, ok)]) == 0
        return bool(ok.item()), Q.cpu().numpy()
    return go


def columns(n, off, seed):
    """Unitary times I + H/2, H Hermitian with entries of random sign up to `off`."""
    rng = np.random.default_rng(seed)
    U, _ = np.linalg.qr(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    H = rng.uniform(-1, 1, (n, n)) + 1j * rng.uniform(-1, 1, (n, n))
    H = H + H.conj().T
    return U @ (np.eye(n) + 0.5 * off * H / np.abs(H).max())


@pytest.mark.parametrize("n", [1, 2, 7, 30, 48, 72])
@pytest.mark.parametrize("off", [1e-7, 3.4e-7, 1e-6, 3e-6, 1e-5, 1e-4, 5e-4])
def test_accepted_means_orthonormal(run, n, off):
    ok, Q = run(columns(n, off, n))
    if ok:
        assert np.abs(Q.conj().T @ Q - np.eye(n)).max() <= 5e-15
    if off <= 3.4e-7:
        assert ok
    if off >= 1e-4 and n > 1:
        assert not ok


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan, 1e30])
def test_unusable_columns_are_refused(run, bad):
    X = columns(24, 1e-7, 1)
    X[3, 5] = bad
    assert not run(X)[0]
