"""The distance form of the design update that k_mma_step runs (mma_box_step) against the update as the rules
state it (mma_box_update), both compiled for the host, over ordinary states and over values far from them:
infinities, NaN, zeros of both signs, huge and tiny gradients and boxes, asymptotes on the wrong side.  The two
differ by rounding only: the distances a, b and the quotient carry a few half-ulps each of quantities no larger
than 10 spans, 20 of them at most, so 20 * 1.2e-16 * 10 spans < 3e-14 spans, plus an ulp of |x| where the box is
small against the value.  Where either gives a NaN or an infinity both do."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1603_06855_gb300", "csrc")
HARNESS = r"""
#include "mma_update.cuh"
extern "C" void run(int which, long long n, const double* x, const double* df, double* a, double* b, double* lo,
                    double* up, double* out, int iter, double xmin, double xmax) {
  for (long long i = 0; i < n; ++i) {
    if (which) mma_box_step(x[i], df[i], iter, xmin, xmax, 1e-5 / (xmax - xmin), a + i, b + i, lo + i, up + i, out + i);
    else mma_box_update(x[i], df[i], iter, xmin, xmax, a + i, b + i, lo + i, up + i, out + i);
  }
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("mma_step")
    src, lib = d / "h.cpp", d / "libh.so"
    src.write_text(HARNESS)
    subprocess.run([cxx, "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)],
                   check=True, capture_output=True)
    so = ctypes.CDLL(str(lib))
    P = ctypes.c_void_p
    so.run.argtypes = [ctypes.c_int, ctypes.c_longlong] + [P] * 7 + [ctypes.c_int, ctypes.c_double, ctypes.c_double]

    def go(which, x, df, a, b, lo, up, it, xmin, xmax):
        v = [np.array(t, dtype=np.float64) for t in (x, df, a, b, lo, up)] + [np.empty(len(x))]
        so.run(which, len(x), *[t.ctypes.data for t in v], it, xmin, xmax)
        return v[6], v[2], v[3], v[4], v[5]  # new x, xo1, xo2, low, upp
    return go


def same(p, q, tol):
    bad = ~(np.isfinite(p) & np.isfinite(q))
    assert np.array_equal(p[bad], q[bad], equal_nan=True)
    assert np.all(np.abs(p[~bad] - q[~bad]) <= tol[~bad])


@pytest.mark.parametrize("it", [0, 1, 2, 7])
@pytest.mark.parametrize("xmin,xmax", [(0.0, 1.0), (-0.5, 2.0), (0.0, 1e-30), (-1e40, 1e40), (1.0, 1.0 + 1e-9),
                                       (0.0, 1e-100), (-1e200, 1e200)])
def test_step_matches_the_rules(run, it, xmin, xmax):
    rng = np.random.default_rng(7 * it + 1)
    span = xmax - xmin
    n = 20000
    x = xmin + span * rng.uniform(0, 1, n)
    df = rng.standard_normal(n) * 10.0 ** rng.uniform(-12, 12, n)
    df[::11] = 0.0
    a = np.clip(x + span * rng.normal(0, 0.2, n), xmin, xmax)
    b = np.clip(a + span * rng.normal(0, 0.2, n), xmin, xmax)
    a[::13], b[::17] = x[::13], a[::17]
    lo, up = a - span * rng.uniform(-0.01, 12, n), a + span * rng.uniform(-0.01, 12, n)
    p, q = (run(w, x, df, a, b, lo, up, it, xmin, xmax) for w in (0, 1))
    tol = 3e-14 * span + 2.3e-16 * np.abs(x)
    for u, v in zip(p, q):
        same(u, v, tol)
    assert np.all((q[0] >= xmin) & (q[0] <= xmax))


@pytest.mark.parametrize("it", [0, 2])
def test_special_values(run, it):
    odd = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, -np.nan, 1e308, -1e308, 1e160, 5e-324, -1e-310, 0.5])
    g = np.array(np.meshgrid(odd, odd, odd, odd, indexing="ij")).reshape(4, -1)
    for order in ((0, 1, 2, 3), (1, 0, 3, 2)):
        x, df, a, lo = g[list(order)]
        b, up = np.full_like(x, 0.25), np.full_like(x, 0.9)
        with np.errstate(all="ignore"):
            p, q = (run(w, x, df, a, b, lo, up, it, 0.0, 1.0) for w in (0, 1))
        for u, v in zip(p, q):
            same(u, v, 3e-14 + 2.3e-16 * np.abs(np.where(np.isfinite(x), x, 0.0)))
