"""The design map's kernels where their branches change: cells of 2^18 elements and just below (the gradient's
extra pass), with and without the octant mirror, ragged axes; projection sharpness at both sides of the
exponential's table range; variables that are not numbers.  Tolerances as for the small cells: densities 1e-14 of
the largest, gradients 1e-13 (the same FP64 sums in another order).  The oracle holds a dense matrix, so the large
cells are compared with the same averages by shifted arrays, which a small cell compares with the oracle."""
import itertools

import numpy as np
import pytest

from oracle import mixed, projection

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class Shifted:
    """Linear-weight average, projection and chain rule, one np.roll per node offset and parity class."""

    def __init__(self, lattice, n, spacing, radius, octant):
        self.n, self.sp, self.octant = n, spacing, octant
        self.nd = tuple(k // spacing for k in n)
        A = mixed.lat.primitive_vectors(lattice)
        self.terms = []
        for p in itertools.product(range(spacing), repeat=3):
            found = []
            for d in itertools.product(range(-3, 4), repeat=3):
                f = (spacing * np.array(d) + 0.5 * spacing - np.array(p) - 0.5) / np.array(n)
                w = radius - min(np.linalg.norm(A @ (f + np.array(s))) for s in itertools.product((-1, 0, 1), repeat=3))
                if w > 0:
                    found.append((d, w))
            tot = sum(w for _, w in found)
            self.terms += [(p, d, w / tot) for d, w in found]

    def expand(self, x):
        if not self.octant:
            return x.reshape(self.nd)
        phi = x.reshape([k // 2 for k in self.nd])
        for ax in range(3):
            phi = np.concatenate([phi, np.flip(phi, ax)], ax)
        return phi

    def forward(self, x, beta):
        phi, mu = self.expand(x), np.zeros(self.n)
        for p, d, w in self.terms:
            mu[tuple(slice(q, None, self.sp) for q in p)] += w * np.roll(phi, [-k for k in d], (0, 1, 2))
        self.dmu = beta * np.exp(-beta * mu) + np.exp(-beta)
        return 1.0 - np.exp(-beta * mu) + mu * np.exp(-beta)

    def backward(self, g):
        v, out = g * self.dmu, np.zeros(self.nd)
        for p, d, w in self.terms:
            out += w * np.roll(v[tuple(slice(q, None, self.sp) for q in p)], d, (0, 1, 2))
        if self.octant:
            for ax in range(3):
                h = self.nd[ax] // 2
                out = out.take(range(h), ax) + np.flip(out, ax).take(range(h), ax)
        return out.ravel()


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_06855_gb300 import binding, build_lib
    build_lib.build()
    binding.load()


def radius(lattice, n, rad):
    return rad * np.linalg.norm(mixed.lat.primitive_vectors(lattice)[:, 0]) / max(n)


@pytest.mark.parametrize("lattice,n,spacing,rad,octant", [("sc", (12, 8, 16), 2, 2.2, True), ("fcc", (9, 8, 7), 1, 1.4, False)])
def test_shifted_arrays_match_the_oracle(lattice, n, spacing, rad, octant):
    r = radius(lattice, n, rad)
    ref, sh = projection.DesignMap(lattice, n, spacing=spacing, radius=r, octant=octant), Shifted(lattice, n, spacing, r, octant)
    rng = np.random.default_rng(3)
    x, g = rng.uniform(0, 1, ref.nvars), rng.standard_normal(n)
    assert np.abs(sh.forward(x, 5.0).reshape(-1) - np.asarray(ref.forward(x, 5.0)).reshape(-1)).max() <= 1e-14
    b = np.asarray(ref.backward(x, 5.0, g)).ravel()
    assert np.abs(sh.backward(g) - b).max() <= 1e-13 * np.abs(b).max()


@pytest.mark.parametrize("lattice,n,spacing,rad,octant", [
    ("sc", (64, 64, 64), 2, 2.2, True), ("sc", (64, 64, 60), 2, 2.2, True), ("fcc", (64, 64, 64), 1, 1.4, False),
    ("bcc", (63, 65, 64), 1, 1.4, False), ("sc", (67, 61, 65), 1, 1.4, False), ("sc", (64, 64, 64), 1, 1.2, True)])
@pytest.mark.parametrize("beta", [0.5, 689.0, 691.0])
def test_large_cells(lattice, n, spacing, rad, octant, beta):
    from paper_1603_06855_gb300.solver import DesignMap
    r = radius(lattice, n, rad)
    sh = Shifted(lattice, n, spacing, r, octant)
    dm = DesignMap(lattice, n, spacing=spacing, radius=r, octant=octant)
    rng = np.random.default_rng(n[1])
    x = rng.uniform(0.0, 1.0, dm.nvars)
    x[::7], x[::11] = 0.0, 1.0
    rho, rho_ref = dm.project(torch.from_numpy(x), beta).cpu().numpy(), sh.forward(x, beta)
    assert np.abs(rho - rho_ref).max() <= 1e-14 * np.abs(rho_ref).max()
    g = rng.standard_normal(n)
    gx, gx_ref = dm.backprop(torch.from_numpy(g)).cpu().numpy(), sh.backward(g)
    assert np.abs(gx - gx_ref).max() <= 1e-13 * np.abs(gx_ref).max()
    dm.close()


def test_variables_outside_the_range_are_clamped():
    from paper_1603_06855_gb300.solver import DesignMap
    dm = DesignMap("sc", (8, 8, 8), spacing=1, radius=0.5 / 8)  # each element sees its own node
    x = torch.full((512,), 0.5, dtype=torch.float64)
    odd = torch.tensor([float("nan"), -float("nan"), float("inf"), -float("inf"), -0.0, -3.0, 7.0, 1.0 + 2e-16])
    x[:8] = odd.to(torch.float64)
    rho = dm.project(x, 4.0).cpu().numpy().ravel()
    e = np.exp(-4.0)
    top = 1.0 - e + e
    want = [0.0, 0.0, top, 0.0, 0.0, 0.0, top, top]
    assert np.abs(rho[:8] - want).max() <= 1e-15
    assert np.abs(rho[8:] - (1.0 - np.exp(-2.0) + 0.5 * e)).max() <= 1e-15
    dm.close()
