"""The adjoint's synthesis and reduction over grids where their loops end unevenly: odd axes (the middle voxel is its
own mirror image), fewer and more columns (j, l) than a warp, more groups of voxel pairs than a CTA has warps, every
cutoff's register shape that a small dense problem allows, one (k, band) pair and many.  All-band gradients against
the oracle's sensitivities at the forms' targets, 1e-5 (FP64) and 1e-4 (mixed) relative L2."""
import numpy as np
import pytest

import workloads as wl
from oracle import mixed, sensitivity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["mixed", "fp64"])
@pytest.mark.parametrize("n,M,nk", [((3, 3, 3), 1, 1), ((37, 4, 5), 1, 3), ((67, 6, 11), 1, 12), ((4, 3, 70), 1, 2),
                                    ((9, 7, 6), 2, 5), ((6, 17, 5), 2, 2), ((9, 8, 7), 3, 1)])
def test_gradient_on_uneven_grids(form, n, M, nk):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_06855_gb300 import binding as B
    from paper_1603_06855_gb300 import build_lib
    from paper_1603_06855_gb300.solver import BandSolver
    build_lib.build()
    rng = np.random.default_rng(n[0] + nk)
    rho = rng.uniform(0.2, 0.9, n)
    Q = rng.uniform(0.05, 0.45, (nk, 3))
    nb = 5
    P = mixed.build("bcc", n, M, rho, wl.TUNGSTEN_CARBIDE, wl.EPOXY, 3.0)
    lam, sols = mixed.bands(P, Q, nb, keep=True)
    w = np.full_like(lam, 1.0 / lam.max())
    ref = sensitivity.weighted(P, sols, w).reshape(n)
    s = BandSolver("bcc", n, M, nb, wl.TUNGSTEN_CARBIDE, wl.EPOXY, Q, penal=3.0, precision=form,
                   tol=1e-4 if form == "mixed" else 0.0)
    s.set_design(torch.from_numpy(rho).cuda())
    s.bands()
    _, g = s.gap_and_grad(mode=B.PC_GRAD_ALLBANDS, weights=torch.from_numpy(w))
    assert np.linalg.norm(g.cpu().numpy() - ref) <= (1e-4 if form == "mixed" else 1e-5) * np.linalg.norm(ref)
    assert s.stats().status == B.PC_OK
    s.close()
