"""The sliced products of the mixed form's final step, slice pair by slice pair.  Operands whose digits (6 bits) lie in one
slice each, i of the operator and j of the column, have a product that is an integer times a power of two: it must
come out exactly for every pair that is kept (i + j <= 9 of eight slices up to N = 1008, i + j <= 11 of ten above) and
as zero for the others.  So no pair, scale, K chunk (two above N = 1008) or column tile can be lost or doubled unseen,
down to the last digit.  Then ordinary operands against FP64 products: both sides round to some 1e-15 of the largest
entry (the ten slices carry more digits than FP64, eight 2e-12), 2e-14 and 1e-10.

Row and column scales are set by an entry of 1 that meets a zero of the other operand; digits of the leading slice are
at most 15, of the others 31."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1603_06855_gb300")
HARNESS = r"""
#include "gemm_tc.h"
extern "C" int run(int N, int ncols, const double2* W, const double2* X, double2* C, int* status) {
  OzPlan* p = oz_plan_create(N, ncols, status, nullptr);
  if (!oz_available(p)) { oz_plan_destroy(p); return 100; }
  // W holds two operators, the second is also passed as the third
  int rc = oz_prepare_operators(p, W, W + (long long)N * N, 1.0, 1.0, 0);
  if (!rc) rc = oz_slice_columns(p, X, ncols, 0, 0);
  for (int g = 0; g < 3 && !rc; ++g) rc = oz_gemm(p, g, 0, ncols, C + (long long)g * ncols * N, 0);
  if (cudaDeviceSynchronize() != cudaSuccess) rc = 101;
  oz_plan_destroy(p);
  return rc;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_06855_gb300 import binding, build_lib
    lib = build_lib.build()
    binding.load()
    nvcc = build_lib._nvcc()
    if shutil.which(nvcc) is None:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("pairs")
    src, out = d / "h.cu", d / "libh.so"
    src.write_text(HARNESS)
    subprocess.run([nvcc, *build_lib.ARCH, *build_lib.FLAGS, "-shared", "-I", os.path.join(PKG, "csrc"), str(src), lib,
                    "-Xlinker", "-rpath", "-Xlinker", PKG, "-o", str(out)], check=True, capture_output=True)
    so = ctypes.CDLL(str(out))

    def go(W, X):
        """C[g][col] = W_g X[col] for g in (0, 1, 1)."""
        N, ncols = W.shape[-1], X.shape[0]
        w, x = (torch.from_numpy(np.ascontiguousarray(t)).cuda() for t in (W, X))
        C = torch.full((3, ncols, N), float("nan"), dtype=torch.complex128, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        P = ctypes.c_void_p
        assert so.run(N, ncols, P(w.data_ptr()), P(x.data_ptr()), P(C.data_ptr()), P(status.data_ptr())) == 0
        assert status.item() == 0
        return C.cpu().numpy()
    return go


def digits(rng, shape, top):
    return rng.integers(-top, top + 1, shape) + 1j * rng.integers(-top, top + 1, shape)


@pytest.mark.parametrize("N,ncols", [(343, 70), (1008, 33), (1009, 33), (1331, 70)])
def test_every_slice_pair_is_exact(run, N, ncols):
    slices, most = (8, 9) if N <= 1008 else (10, 11)
    rng = np.random.default_rng(N)
    unit = lambda i: 4.0 * 2.0 ** (-6 * i)  # noqa: E731  (a row whose largest entry is 1 has scale 4)
    j = np.arange(ncols) % slices + 1
    top = np.where(j == 1, 15, 31)[:, None]
    xd = np.clip(digits(rng, (ncols, N), 31).real, -top, top) + 1j * np.clip(digits(rng, (ncols, N), 31).real, -top, top)
    xd[:, :2] = 0
    X = xd * unit(j)[:, None]
    X[:, 1] = 1.0
    for i in range(1, slices + 1, 2):
        ii = (i, min(i + 1, slices))
        wd = np.stack([digits(rng, (N, N), 15 if i == 1 else 31), digits(rng, (N, N), 31)])
        wd[:, :, :2] = 0
        W = wd * np.array([unit(k) for k in ii])[:, None, None]
        W[:, :, 0] = 1.0
        C = run(W, X)
        for g, h in ((0, 0), (1, 1), (2, 1)):
            want = (xd @ wd[h].T) * (unit(ii[h]) * unit(j))[:, None]  # integers below 2^24: exact
            want[ii[h] + j > most] = 0
            assert np.array_equal(C[g], want), (i, g)


@pytest.mark.parametrize("N,ncols,tol", [(1008, 40, 1e-10), (1009, 65, 2e-14), (1331, 33, 2e-14), (1331, 300, 2e-14)])
def test_ordinary_operands(run, N, ncols, tol):
    rng = np.random.default_rng(N + ncols)
    W = rng.standard_normal((2, N, N)) + 1j * rng.standard_normal((2, N, N))
    W *= 2.0 ** rng.integers(-4, 5, (1, N, 1))
    X = rng.standard_normal((ncols, N)) + 1j * rng.standard_normal((ncols, N))
    C = run(W, X)
    for g, h in ((0, 0), (1, 1), (2, 1)):
        want = X @ W[h].T
        assert np.abs(C[g] - want).max() <= tol * np.abs(want).max()
