"""Uniform cells, where an optimisation starts: the mixed form with several start blocks against the closed form (two
transverse waves and a longitudinal one at every |K|), within the form's 1e-6 and its residual target, in the two dozen
iterations that such a cell takes.  High multiplicities, wide blocks and the Gamma point among the wavevectors."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def closed_form(lattice, M, Q, nb, m):
    from oracle import lattice as lat
    T = np.linalg.inv(lat.primitive_vectors(lattice)).T  # reciprocal vectors by columns, without 2 pi
    g = np.array([(i, j, k) for i in range(-M, M + 1) for j in range(-M, M + 1) for k in range(-M, M + 1)])
    K = 2 * np.pi * np.linalg.norm((Q[:, None, :] + g) @ T.T, axis=2)
    cl = np.sqrt(m["E"] * (1 - m["nu"]) / ((1 + m["nu"]) * (1 - 2 * m["nu"]) * m["rho"]))
    ct = np.sqrt(m["E"] / (2 * (1 + m["nu"]) * m["rho"]))
    return np.sort(np.concatenate([cl * K, ct * K, ct * K], axis=1), axis=1)[:, :nb]


@pytest.mark.parametrize("lattice,M,n,nb,nk,tol,most", [("sc", 2, (5, 11, 9), 21, 40, 0.0, 30), ("fcc", 2, (8, 9, 8), 16, 30, 0.0, 35),
                                                   ("bcc", 2, (9, 8, 7), 20, 20, 1e-4, 35)])
def test_start_blocks(lattice, M, n, nb, nk, tol, most, monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_06855_gb300 import binding as B
    from paper_1603_06855_gb300 import build_lib
    from paper_1603_06855_gb300.solver import BandSolver
    build_lib.build()
    Q = np.random.default_rng(5).uniform(-0.5, 0.5, (nk, 3))
    Q[0] = 0.0
    want = closed_form(lattice, M, Q, nb, wl.TUNGSTEN_CARBIDE)
    zero = want <= 1e-9 * want.max()  # a zero mode's frequency is the root of rounding: its square counts
    for seed in range(12):
        monkeypatch.setenv("PC_INIT_SEED", str(seed))
        s = BandSolver(lattice, n, M, nb, wl.TUNGSTEN_CARBIDE, wl.EPOXY, Q, penal=3.0, precision="mixed", tol=tol)
        s.set_design(torch.ones(n, dtype=torch.float64, device="cuda"))
        om = s.bands().cpu().numpy()
        st = s.stats()
        s.close()
        assert st.status == B.PC_OK
        assert np.all(om[zero] ** 2 <= 1e-9 * want.max() ** 2)
        assert np.abs(om[~zero] / want[~zero] - 1.0).max() <= 1e-6, seed
        assert st.iterations <= most, seed
