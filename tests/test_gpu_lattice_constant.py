"""The lattice constant only sets the units: relative gaps and their gradients are the same at every size of the cell, from
nanometres to kilometres, and eigenvalues and their gradients scale as a^-2.  To the mixed form's 1e-4 (its
iteration is nondimensional, but rounds differently where the scales are not powers of two), FP64 1e-9."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form,tol", [("mixed", 1e-4), ("fp64", 1e-9)])
def test_gradients_at_any_size(form, tol):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_06855_gb300 import binding as B
    from paper_1603_06855_gb300 import build_lib
    from paper_1603_06855_gb300.solver import BandSolver
    build_lib.build()
    rng = np.random.default_rng(8)
    n, nk, nb = (9, 8, 10), 5, 6
    Q = rng.uniform(-0.5, 0.5, (nk, 3))
    rho = torch.from_numpy(wl.random_design(n, rng)).cuda()
    w = torch.from_numpy(rng.uniform(0.5, 1.5, (nk, nb)) * 1e-9).cuda()
    first = None
    for a in (1.0, 1e-9, 3e-6, 1e-3, 0.02, 50.0, 1e3):
        s = BandSolver("fcc", n, 2, nb, wl.TUNGSTEN_CARBIDE, wl.EPOXY, Q, penal=3.0, precision=form, a=a,
                       tol=1e-5 if form == "mixed" else 1e-11)
        s.set_design(rho)
        s.bands()
        got = [s.gap_and_grad(n_lower=3)[1], s.gap_ks_and_grad(3, 20.0)[1],
               s.gap_and_grad(mode=B.PC_GRAD_ALLBANDS, weights=w)[1] * a * a]
        got = [t.clone() for t in got]
        assert s.stats().status == B.PC_OK
        s.close()
        first = first or got
        for x, y in zip(first, got):
            assert torch.linalg.norm(x - y) <= tol * torch.linalg.norm(x), a
