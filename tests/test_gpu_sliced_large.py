"""The mixed form's final Rayleigh-Ritz step at M = 5 (N = 1331): its operator products run as ten-slice
products with K in two chunks and 32 columns a tile.  Against the FP64 form (whose products are FP64
GEMMs) on the same design, for column counts around the tile: frequencies 1e-7 (the mixed form's error is
second order in its residual target, 1e-4, on these few separated bands; its bound is 1e-6) and the
eigenvectors' Omega-normalisation exported from the step, 1e-9."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nk,nb", [(1, 1), (1, 4), (2, 5)])
def test_sliced_products_above_1008(nk, nb):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_06855_gb300 import binding as B, build_lib
    from paper_1603_06855_gb300.solver import BandSolver
    build_lib.build()
    B.load()
    n = (11, 13, 12)
    rho = torch.from_numpy(wl.random_design(n, np.random.default_rng(55))).cuda()
    Q = np.array([[0.11, 0.23, 0.41], [0.37, -0.2, 0.05]])[:nk]
    om, vec = {}, None
    for form in ("mixed", "fp64"):
        s = BandSolver("bcc", n, 5, nb, wl.TUNGSTEN_CARBIDE, wl.EPOXY, Q, penal=3.0, precision=form,
                       tol=1e-4 if form == "mixed" else 1e-8)
        s.set_design(rho)
        om[form] = s.bands().cpu().numpy()
        st = s.stats()
        assert st.status == B.PC_OK
        if form == "mixed":
            assert st.rr_sliced == 1
            N = st.N
            vec = s.export(B.PC_EXPORT_EIGVEC).view(np.complex128).reshape(nk, nb, 3, N)
            T = s.export(B.PC_EXPORT_TOEP).view(np.complex128).reshape(3, N, N)[0]
        s.close()
    assert np.abs(om["mixed"] / om["fp64"] - 1.0).max() <= 1e-7
    for k in range(nk):
        G = np.einsum("acp,pq,bcq->ab", vec[k].conj(), T, vec[k], optimize=True)
        assert np.abs(G - np.eye(nb)).max() <= 1e-9
