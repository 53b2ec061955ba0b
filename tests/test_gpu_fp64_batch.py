"""FP64 designs side by side: a batch's designs give the bits that each gives alone, although alone its projected
problems get a cluster of CTAs each and among others one CTA."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("designs,workers", [(12, 12), (3, 2)])
def test_batch_of_reference_solves(designs, workers):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_06855_gb300 import binding as B
    from paper_1603_06855_gb300 import build_lib
    from paper_1603_06855_gb300.solver import BandSolver, BatchSolver
    build_lib.build()
    rng = np.random.default_rng(designs)
    n = (7, 8, 6)
    cells = [wl.Workload("cell", lat, n, 1, nb, rng.uniform(-0.5, 0.5, (4, 3)), wl.random_design(n, rng), 3.0, (2,), 0)
             for lat, nb, _ in zip(["sc", "bcc", "fcc"] * designs, [5, 9, 12] * designs, range(designs))]
    bs = BatchSolver(cells, precision="fp64", workers=workers)
    bs.set_designs([torch.from_numpy(w.rho) for w in cells])
    together = [o.clone() for o in bs.bands()]
    torch.cuda.synchronize()
    for i, w in enumerate(cells):
        assert bs.stats(i).status == B.PC_OK
        s = BandSolver.from_workload(w, precision="fp64")
        s.set_design(torch.from_numpy(w.rho).cuda())
        assert torch.equal(s.bands(), together[i])
        s.close()
    bs.close()
