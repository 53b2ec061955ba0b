"""The FP64 projected problems on both sides of the rule that gives each a cluster of CTAs (8 per problem while the
chip has as many SMs: 19 problems on 152), over block widths whose products split unevenly among the CTAs.
Frequencies against the oracle at the FP64 form's target, 1e-9."""
import numpy as np
import pytest

import workloads as wl
from oracle import mixed

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [1, 5, 20])
@pytest.mark.parametrize("nk", [1, 18, 19, 20, 38])
def test_few_and_many_problems(nb, nk):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_06855_gb300 import binding as B
    from paper_1603_06855_gb300 import build_lib
    from paper_1603_06855_gb300.solver import BandSolver
    build_lib.build()
    n = (5, 6, 7)
    rng = np.random.default_rng(nk)
    rho = wl.random_design(n, rng)
    Q = rng.uniform(-0.5, 0.5, (nk, 3))
    lam = np.asarray(mixed.bands(mixed.build("fcc", n, 1, rho, wl.TUNGSTEN_CARBIDE, wl.EPOXY, 3.0), Q, nb))
    s = BandSolver("fcc", n, 1, nb, wl.TUNGSTEN_CARBIDE, wl.EPOXY, Q, penal=3.0, precision="fp64")
    s.set_design(torch.from_numpy(rho).cuda())
    om = s.bands().cpu().numpy()
    assert s.stats().status == B.PC_OK
    assert np.abs(om / np.sqrt(lam) - 1.0).max() <= 1e-9
    s.close()
