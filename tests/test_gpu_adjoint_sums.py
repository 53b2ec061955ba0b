"""The adjoint's weighted sums where a chunk of (k, band) pairs is cut, left out or one of many: all 2600 pairs of 130
k-points and 20 bands, single pairs in the first, a middle and the last chunk, and none, on a small cell (many
chunks at once) and on a 72 x 73 x 71 one (one chunk fills the chip).  The FP64 form's kernels are compared with the sum of
their own gradients over single k-points, which is linear in the weights: 1e-12; the mixed form's FP32 sums with the
FP64 form's gradient of the same bands, at the form's target, 1e-4."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(5, 6, 7), (72, 73, 71)])
def test_pairs_over_all_chunks(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_06855_gb300 import binding as B
    from paper_1603_06855_gb300 import build_lib
    from paper_1603_06855_gb300.solver import BandSolver
    build_lib.build()
    rng = np.random.default_rng(n[0])
    nk, nb = 130, 20
    Q = rng.uniform(-0.5, 0.5, (nk, 3))
    rho = torch.from_numpy(rng.uniform(0.2, 0.9, n)).cuda()
    grads = {}
    full = torch.from_numpy(rng.uniform(0.5, 1.5, (nk, nb)) * 1e-9).cuda()
    for form in ("fp64", "mixed"):
        s = BandSolver("sc", n, 1, nb, wl.TUNGSTEN_CARBIDE, wl.EPOXY, Q, penal=3.0, precision=form,
                       tol=1e-5 if form == "mixed" else 1e-9)
        s.set_design(rho)
        s.bands()

        def grad(w):
            return s.gap_and_grad(mode=B.PC_GRAD_ALLBANDS, weights=w)[1].clone()

        grads[form] = grad(full)
        if form == "fp64":
            parts = torch.zeros_like(grads[form])
            for k in range(nk):
                w = torch.zeros_like(full)
                w[k] = full[k]
                parts += grad(w)
            assert torch.linalg.norm(parts - grads[form]) <= 1e-12 * torch.linalg.norm(parts)
        assert torch.count_nonzero(grad(torch.zeros_like(full))) == 0
        s.close()
    assert torch.linalg.norm(grads["mixed"] - grads["fp64"]) <= 1e-4 * torch.linalg.norm(grads["fp64"])
