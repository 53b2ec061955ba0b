"""K-point sets of more projected problems than one launch takes (sixteen per SM): frequencies against the oracle across
the launches' edges, 1e-9 (FP64) and 1e-6 (mixed), the forms' targets; and the device memory that a k-point of the
widest block costs, which the scratch of those problems must not be part of.  The arrays kept per k-point come to
2.08 MB (FP64, 24 columns, N = 27) and 1.73 MB (mixed, 23 columns); a tenth is left for rounding up."""
import numpy as np
import pytest

import workloads as wl
from oracle import mixed

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def solver():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_06855_gb300 import build_lib
    from paper_1603_06855_gb300.solver import BandSolver
    build_lib.build()

    def make(form, n, nb, Q):
        return BandSolver("bcc", n, 1, nb, wl.TUNGSTEN_CARBIDE, wl.EPOXY, Q, penal=3.0, precision=form,
                          tol=1e-4 if form == "mixed" else 0.0)
    return make


@pytest.mark.parametrize("form,nk", [("fp64", 2600), ("mixed", 5200)])
def test_more_problems_than_a_launch(solver, form, nk):
    from paper_1603_06855_gb300 import binding as B
    n, nb = (4, 5, 3), 3
    rng = np.random.default_rng(nk)
    rho, Q = wl.random_design(n, rng), rng.uniform(-0.5, 0.5, (nk, 3))
    at = np.unique(np.clip(np.concatenate([np.arange(nk // 100) * 100] + [e + np.arange(-2, 3) for e in (2432, 2600, 5032, nk)]),
                           0, nk - 1))
    P = mixed.build("bcc", n, 1, rho, wl.TUNGSTEN_CARBIDE, wl.EPOXY, 3.0)
    lam = np.asarray(mixed.bands(P, Q[at], nb))
    s = solver(form, n, nb, Q)
    s.set_design(torch.from_numpy(rho).cuda())
    om = s.bands().cpu().numpy()
    assert s.stats().status == B.PC_OK
    assert np.abs(om[at] / np.sqrt(lam) - 1.0).max() <= (1e-9 if form == "fp64" else 1e-6)
    s.close()


@pytest.mark.parametrize("form,most", [("fp64", 2.3e6), ("mixed", 1.95e6)])
def test_memory_per_kpoint(solver, form, most):
    used = []
    for nk in (5000, 7000):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        s = solver(form, (3, 3, 3), 20, np.random.default_rng(nk).uniform(-0.5, 0.5, (nk, 3)))
        used.append(before - torch.cuda.mem_get_info()[0])
        s.close()
    assert (used[1] - used[0]) / 2000 <= most
