"""The inverse compliance operators of cells with strong contrast (modulus ratios of 1e3 to 3e4, stiff cubes in a soft
matrix and the reverse, grids as small as the cutoff allows): T W - 1 entry by entry against what a stable inversion
leaves, N eps cond(T), and W Hermitian."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,M,n", [("sc", 1, (4, 5, 3)), ("fcc", 2, (6, 8, 9)), ("bcc", 2, (5, 5, 5)), ("bcc", 3, (7, 11, 10)),
                                         ("bcc", 3, (11, 11, 8)), ("sc", 4, (9, 10, 9))])
@pytest.mark.parametrize("ratio", [1e-3, 6e-5, 3e-5])
@pytest.mark.parametrize("stiff", [0, 1])
def test_residual_of_the_inverse(lattice, M, n, ratio, stiff):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_06855_gb300 import binding as B
    from paper_1603_06855_gb300 import build_lib
    from paper_1603_06855_gb300.solver import BandSolver
    build_lib.build()
    hard, soft = dict(wl.TUNGSTEN_CARBIDE), dict(wl.EPOXY)
    soft["E"] = hard["E"] * ratio
    rho = np.full(n, 1.0 - stiff)
    rho[tuple(slice(k // 4, 3 * k // 4) for k in n)] = stiff
    s = BandSolver(lattice, n, M, 1, hard, soft, np.array([[0.1, 0.2, 0.3]]), penal=1.0, precision="fp64")
    s.set_design(torch.from_numpy(rho).cuda())
    N = (2 * M + 1) ** 3
    T = s.export(B.PC_EXPORT_TOEP).view(np.complex128).reshape(3, N, N)[1:]
    W = s.export(B.PC_EXPORT_WINV).view(np.complex128).reshape(2, N, N)
    s.close()
    for t, w in zip(T, W):
        ev = np.linalg.eigvalsh(t)
        assert np.abs(t @ w - np.eye(N)).max() <= N * np.finfo(float).eps * ev[-1] / ev[0]
        assert np.array_equal(np.triu(w, 1), np.tril(w, -1).conj().T)
