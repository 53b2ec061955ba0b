"""The iteration cap at the edge of the residual target.  The block iteration aims below the tolerance and gives a
k-point that has met it one more iteration to get there, but the tolerance is what a call promises: where the
last check before the cap finds the residual a little below the tolerance, the call has converged
(PC_OK, no k-point counted as unconverged), and one check earlier, above the tolerance, it has not.  The residual of
every check is read from the library's debug output; tolerances an eighth of a decade apart, of which the
residuals' steps (a factor of two to four an iteration) leave a quarter or more in that window."""
import re

import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form,decade", [("fp64", -6), ("mixed", -2)])
def test_tolerance_met_at_the_cap(form, decade, monkeypatch, capfd):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_06855_gb300 import binding as B
    from paper_1603_06855_gb300 import build_lib
    from paper_1603_06855_gb300.solver import BandSolver
    build_lib.build()
    n = (8, 9, 7)
    rho = torch.from_numpy(wl.random_design(n, np.random.default_rng(12))).cuda()
    monkeypatch.setenv("PC_DEBUG", "1")

    def call(tol, cap):
        s = BandSolver("sc", n, 2, 6, wl.TUNGSTEN_CARBIDE, wl.EPOXY, np.array([[0.21, 0.13, 0.37]]), penal=3.0,
                       precision=form, tol=tol, max_iter=cap)
        s.set_design(rho)
        capfd.readouterr()
        s.bands()
        res = [float(v) for v in re.findall(r"max_res (\S+) at k \d+; open", capfd.readouterr().err)]
        st = s.stats()
        s.close()
        return st, res

    found = 0
    for j in range(8):
        tol = 10.0 ** (decade - j / 8)
        st, res = call(tol, 0)
        assert st.status == B.PC_OK and st.unconverged_k == 0
        at = next(i for i, r in enumerate(res) if r <= tol)
        if not 0.51 * tol < res[at] < 0.99 * tol or at == 0:
            continue
        found += 1
        st, _ = call(tol, at + 1)  # checks 0 .. at
        assert (st.status, st.unconverged_k, st.iterations) == (B.PC_OK, 0, at + 1)
        st, _ = call(tol, at)
        assert (st.status, st.unconverged_k, st.iterations) == (B.PC_ENOCONV, 1, at)
    assert found >= 1
