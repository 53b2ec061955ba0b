"""GPU parity of both forms where the k-points and columns of one call converge at different iterations:
the later iterations cover the open k-points and unconverged columns only, through lists that are
compacted 256 k-points at a time.  One k-point, the edges of a chunk and several chunks in each of the
mixed form's k groups; wavevectors from near the zone centre to its boundary, so that neither the first
nor the last of the list converges last.  Tolerances are the forms' targets: frequencies 1e-6 (mixed)
and 1e-9 (FP64)."""
import numpy as np
import pytest

import workloads as wl
from oracle import mixed

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["mixed", "fp64"])
@pytest.mark.parametrize("nk", [1, 2, 255, 256, 257, 530])
def test_many_kpoints_match_the_oracle(form, nk):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_06855_gb300 import binding as B
    from paper_1603_06855_gb300 import build_lib
    from paper_1603_06855_gb300.solver import BandSolver
    build_lib.build()
    n, nb = (6, 6, 6), 4
    rng = np.random.default_rng(5)
    rho = wl.random_design(n, rng)
    Q = rng.uniform(-0.5, 0.5, (nk, 3)) * rng.choice([0.05, 0.3, 1.0], (nk, 1))
    P = mixed.build("sc", n, 1, rho, wl.TUNGSTEN_CARBIDE, wl.EPOXY, 3.0)
    lam = np.asarray(mixed.bands(P, Q, nb))[:, :nb]
    s = BandSolver("sc", n, 1, nb, wl.TUNGSTEN_CARBIDE, wl.EPOXY, Q, penal=3.0, precision=form,
                   tol=1e-4 if form == "mixed" else 0.0)
    s.set_design(torch.from_numpy(rho).cuda())
    om = s.bands().cpu().numpy()
    assert s.stats().status == B.PC_OK
    assert np.abs(om / np.sqrt(lam) - 1.0).max() <= (1e-6 if form == "mixed" else 1e-9)
    s.close()
