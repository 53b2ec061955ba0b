"""GPU parity of both forms across block widths: the projected problems of the iteration have
n = 3 (bands + 3) columns in the mixed form and 3 (bands + 4) in the FP64 form (at most 72), and their
kernels change shape with n (planes per lane of the eigenvector replay at n = 32 and 64, odd and even
counts, partial panels, two tiles per thread above n = 56, the largest 72).  Tolerances are the forms'
targets: frequencies 1e-6 and all-band gradients 1e-4 (mixed), 1e-9 and 1e-5 (FP64)."""
import numpy as np
import pytest

import workloads as wl
from oracle import mixed, sensitivity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cell():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_06855_gb300 import binding, build_lib
    build_lib.build()
    binding.load()
    n = (7, 5, 6)
    rho = wl.random_design(n, np.random.default_rng(31))
    Q = np.array([[0.11, 0.23, 0.41], [0.5, 0.5, 0.0], [0.37, -0.2, 0.05]])
    P = mixed.build("fcc", n, 1, rho, wl.TUNGSTEN_CARBIDE, wl.EPOXY, 3.0)
    lam, sols = mixed.bands(P, Q, 21, keep=True)
    return n, rho, Q, P, lam, sols


@pytest.mark.parametrize("form,nb", [("mixed", nb) for nb in (1, 2, 6, 7, 8, 9, 18, 19, 20, 21)]
                         + [("fp64", nb) for nb in (1, 6, 7, 14, 15, 17, 20, 21)])
def test_block_widths(cell, form, nb):
    from paper_1603_06855_gb300 import binding as B
    from paper_1603_06855_gb300.solver import BandSolver
    n, rho, Q, P, lam, sols = cell
    s = BandSolver("fcc", n, 1, nb, wl.TUNGSTEN_CARBIDE, wl.EPOXY, Q, penal=3.0, precision=form,
                   tol=1e-4 if form == "mixed" else 0.0)
    tol_w, tol_g = (1e-6, 1e-4) if form == "mixed" else (1e-9, 1e-5)
    s.set_design(torch.from_numpy(rho).cuda())
    om = s.bands().cpu().numpy()
    ref = np.sqrt(lam[:, :nb])
    assert np.abs(om / ref - 1.0).max() <= tol_w
    w = np.zeros_like(lam)
    w[:, :nb] = 1.0 / lam.max()
    _, g = s.gap_and_grad(mode=B.PC_GRAD_ALLBANDS, weights=torch.from_numpy(w[:, :nb].copy()))
    g_ref = sensitivity.weighted(P, sols, w).reshape(n)
    assert np.linalg.norm(g.cpu().numpy() - g_ref) <= tol_g * np.linalg.norm(g_ref)
    assert s.stats().status == B.PC_OK
    s.close()
