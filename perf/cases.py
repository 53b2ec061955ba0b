"""The work this library is used for, as timed cases.

Kinds of case (``case["kind"]``):

* ``step``   one evaluation of a design inside an optimisation: densities from the program's own
  single-precision parameters, the operators of the design, the lowest bands at every wavevector,
  a weighted sum of eigenvalues and its gradient, carried back to the parameters.  The mixed form;
  such a program keeps single precision, which holds what the form promises (frequencies to about
  1e-8, gradients to about 1e-5), and asks for the residual target (1e-4) that gradients want.
* ``fp64``   the same evaluation in the FP64 form: the reference a program checks itself against,
  in double precision throughout, on a shifted grid of wavevectors (zone averages), solved to a
  residual of 1e-11.
* ``scan``   many small cells in one call: band structures and gaps of sphere inclusions over
  lattices and volume fractions (the volume-fraction scans), no gradient.
* ``apply``  the operators of a new design applied to given vectors at one wavevector: what a
  program with its own eigensolver, or a residual check, asks for.
* ``map``    the design parametrisation around the solver: reduced field -> densities, the
  gradient back, and one update of the design variables.

Sizes are those of the workloads (8^3 to 32^3 voxels, cutoffs 1 to 4, 10 to 100 wavevectors), of
the uneven batch (cutoffs up to 5) and of the 48^3 cell that designs are published on.
"""
import math

import numpy as np
import torch

import workloads as wl
from paper_1603_06855_gb300 import binding as B
from paper_1603_06855_gb300.solver import MMA, BandSolver, BatchSolver, DesignMap

DEV = "cuda"
PENAL = 3.0   # exponent of the density law, as in the workloads
BETA = 4.0    # sharpness of the projection, two doublings into its continuation


def listed():
    return [
        # between two solves of an optimisation at 48^3: project, chain rule, update (SC octant)
        {"name": "map_sc48_octant", "kind": "map", "lattice": "sc", "n0": 48, "n1": 48, "n2": 48, "spacing": 2, "octant": True},
        # the same on a larger cell without symmetry, a variable on every voxel
        {"name": "map_fcc96_full", "kind": "map", "lattice": "fcc", "n0": 96, "n1": 96, "n2": 96, "spacing": 1, "octant": False},
        # the smallest whole evaluation: the binary-cube cell's size in the FP64 form
        {"name": "fp64_sc8_M1", "kind": "fp64", "lattice": "sc", "n0": 8, "n1": 8, "n2": 8, "M": 1, "bands": 6, "grid": 3},
        # a reference solve of the random-field cell's size
        {"name": "fp64_sc16_M2", "kind": "fp64", "lattice": "sc", "n0": 16, "n1": 16, "n2": 16, "M": 2, "bands": 12, "grid": 2},
        # design steps: the random-field cells' sizes, ragged grid and cutoff on the third
        {"name": "step_sc16_M2", "kind": "step", "lattice": "sc", "n0": 16, "n1": 16, "n2": 16, "M": 2, "bands": 12, "nk": 30, "design": "field"},
        {"name": "step_bcc24_M3", "kind": "step", "lattice": "bcc", "n0": 24, "n1": 24, "n2": 24, "M": 3, "bands": 16, "nk": 64, "design": "field"},
        {"name": "step_sc48_M3", "kind": "step", "lattice": "sc", "n0": 48, "n1": 48, "n2": 48, "M": 3, "bands": 9, "nk": 80, "design": "field"},
        # the headline workload: size and kind of design (near-binary, slow to converge)
        {"name": "step_fcc32_M4", "kind": "step", "lattice": "fcc", "n0": 32, "n1": 32, "n2": 32, "M": 4, "bands": 20, "nk": 100, "design": "levelset"},
        # the uneven batch's largest cutoff
        {"name": "step_bcc28_M5", "kind": "step", "lattice": "bcc", "n0": 28, "n1": 25, "n2": 27, "M": 5, "bands": 20, "nk": 24, "design": "field"},
        # a volume-fraction scan: three lattices, three spheres each
        {"name": "scan_spheres_M3", "kind": "scan", "n0": 24, "M": 3, "bands": 8, "nk": 31, "designs": 9},
        # a new design's operators on 48 vectors, in both forms
        {"name": "apply_fp64_M3", "kind": "apply", "lattice": "bcc", "n0": 24, "n1": 24, "n2": 24, "M": 3, "form": "fp64", "cols": 48},
        {"name": "apply_mixed_M4", "kind": "apply", "lattice": "fcc", "n0": 32, "n1": 32, "n2": 32, "M": 4, "form": "mixed", "cols": 240},
    ]


def _axis(rng, M, top):
    """A grid length the cutoff allows, spread over its logarithm, odd ones among them."""
    lo = 2 * M + 2
    return min(top, int(round(math.exp(rng.uniform(math.log(lo), math.log(top + 0.49))))))


def draw(rng):
    kind = rng.choice(["map", "fp64", "step", "step", "step", "scan", "apply", "apply"])
    lattice = rng.choice(["sc", "bcc", "fcc"])
    if kind == "map":
        octant = lattice == "sc" and rng.random() < 0.5
        spacing = rng.choice([1, 2])
        unit = spacing * (2 if octant else 1)
        n = unit * max(8 // unit, int(math.exp(rng.uniform(math.log(8), math.log(96))) / unit))
        return {"kind": kind, "lattice": lattice, "n0": n, "n1": n, "n2": n, "spacing": spacing, "octant": octant}
    if kind == "fp64":
        M = rng.choice([1, 1, 2])
        n = [_axis(rng, M, 20) for _ in range(3)]
        return {"kind": kind, "lattice": lattice, "n0": n[0], "n1": n[1], "n2": n[2], "M": M,
                "bands": rng.randint(4, 12), "grid": rng.choice([2, 2, 3])}
    if kind == "step":
        M = rng.choice([2, 3, 3, 4, 4])
        n = [_axis(rng, M, 48 if M < 4 else 32) for _ in range(3)]
        nk = int(round(math.exp(rng.uniform(math.log(13), math.log(100)))))
        return {"kind": kind, "lattice": lattice, "n0": n[0], "n1": n[1], "n2": n[2], "M": M,
                "bands": rng.randint(6, 20), "nk": nk,
                "design": rng.choice(["field", "field", "levelset"]) if M > 2 else "field"}
    if kind == "scan":
        M = rng.choice([2, 3])
        return {"kind": kind, "n0": _axis(rng, M, 32), "M": M, "bands": rng.randint(7, 10),
                "nk": rng.randint(13, 31), "designs": 3 * rng.randint(1, 3)}
    M = rng.choice([1, 2, 3, 4])
    n = [_axis(rng, M, 40) for _ in range(3)]
    form = rng.choice(["fp64", "mixed"])
    top = 240 if form == "mixed" else 64
    cols = int(round(math.exp(rng.uniform(math.log(8), math.log(top)))))
    return {"kind": kind, "lattice": lattice, "n0": n[0], "n1": n[1], "n2": n[2], "M": M, "form": form, "cols": cols}


# ---------------------------------------------------------------------------
# inputs

def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _field(n, gen):
    """Periodic Gaussian random field (correlation length a sixth of the cell), as the workloads'."""
    w = torch.randn(n, generator=gen, device=DEV, dtype=torch.float64)
    kern = 1.0
    for ax, k in enumerate(n):
        d = (torch.arange(k, device=DEV, dtype=torch.float64) / k + 0.5) % 1.0 - 0.5
        shape = [1, 1, 1]
        shape[ax] = k
        kern = kern * torch.exp(-18.0 * d * d).reshape(shape)
    z = torch.fft.ifftn(torch.fft.fftn(w) * torch.fft.fftn(kern)).real
    return (z - z.mean()) / z.std()


def _levelset(n, gen):
    """Smooth single-network inclusion as the headline workload's: eight cosines with |m| <= 2, about
    their median, slope 8 deviations (the logit of the density)."""
    m = torch.randint(-2, 3, (8, 3), generator=gen, device=DEV).to(torch.float64)
    m[:, 0] += (m.abs().sum(1) == 0).to(torch.float64)
    a = torch.randn(8, generator=gen, device=DEV, dtype=torch.float64)
    ph = 2 * math.pi * torch.rand(8, generator=gen, device=DEV, dtype=torch.float64)
    g = torch.meshgrid(*[(torch.arange(k, device=DEV, dtype=torch.float64) + 0.5) / k for k in n], indexing="ij")
    phi = sum(a[j] * torch.cos(2 * math.pi * (m[j, 0] * g[0] + m[j, 1] * g[1] + m[j, 2] * g[2]) + ph[j]) for j in range(8))
    return 8.0 * (phi - phi.median()) / phi.std()


def _shifted_grid(g):
    """Shifted g x g x g zone grid, one of each pair k, -k (their bands are equal)."""
    pts = [((i + 0.5) / g, (j + 0.5) / g, (l + 0.5) / g) for i in range(g) for j in range(g) for l in range(g)]
    return np.array([p for p in pts if p <= tuple(1.0 - c for c in p)])


def _grid_of(case):
    return (case["n0"], case["n1"], case["n2"])


def _spheres(case, seed):
    """The scan's cells: SC, BCC, FCC in turn, volume fractions 0.30 to 0.60 moved by the seed."""
    r = np.random.default_rng(seed)
    out = []
    for i in range(case["designs"]):
        lat = ("sc", "bcc", "fcc")[i % 3]
        vf = 0.30 + 0.10 * (i // 3) + float(r.uniform(0.0, 0.1))
        rho = wl.sphere_inclusion(lat, (case["n0"],) * 3, vf, sub=2)
        out.append(wl.Workload("sphere", lat, (case["n0"],) * 3, case["M"], case["bands"], wl.kpath(lat, case["nk"]),
                               rho, 1.0, (6,), 0, 1.0, dict(wl.PAPER_WC), dict(wl.PAPER_EPOXY)))
    return out


def _weights(nk, nb):
    """Equal positive weights on every band, in units of the phases' scale (2 pi)^2 E / rho."""
    lref = (2 * math.pi) ** 2 * wl.EPOXY["E"] / wl.EPOXY["rho"]
    return torch.full((nk, nb), 1.0 / (nk * nb * lref), dtype=torch.float64, device=DEV)


def _inputs(case, seed):
    """The tensors of a pass, from the seed alone."""
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "scan":
        return {"cells": _spheres(case, seed)}
    n = _grid_of(case)
    if kind == "map":
        nv = n[0] * n[1] * n[2] // case["spacing"] ** 3 // (8 if case["octant"] else 1)
        x = torch.rand(nv, generator=gen, device=DEV, dtype=torch.float64)
        noise = torch.randn((2, nv), generator=gen, device=DEV, dtype=torch.float64)
        return {"x": x, "g": torch.randn(n, generator=gen, device=DEV, dtype=torch.float64),
                "x1": (x + 0.1 * noise[0]).clamp(0, 1), "x2": (x + 0.1 * (noise[0] + noise[1])).clamp(0, 1)}
    z = _levelset(n, gen) if case.get("design") == "levelset" else _field(n, gen)
    if kind == "step":
        return {"theta": z.to(torch.float32), "Q": wl.kpath(case["lattice"], case["nk"])}
    if kind == "fp64":
        return {"rho": torch.sigmoid(z), "Q": _shifted_grid(case["grid"])}
    N = (2 * case["M"] + 1) ** 3
    nk = -(-case["cols"] // min(N, _apply_bands(N) + 3))
    Q = np.array([[0.13 + 0.3 * i / nk, 0.21, 0.37 - 0.2 * i / nk] for i in range(nk)])
    v = torch.randn((case["cols"], 3 * N, 2), generator=gen, device=DEV, dtype=torch.float64)
    return {"rho": torch.sigmoid(z), "Q": Q,
            "x": torch.view_as_complex(v if case["form"] == "fp64" else v.to(torch.float32))}


def _apply_bands(N):
    return min(20, N)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(_inputs(case, seed), kind=kind)
    if kind == "map":
        st["map"] = DesignMap(case["lattice"], _grid_of(case), spacing=case["spacing"], octant=case["octant"])
        st["opt"] = MMA(st["map"].nvars, device=DEV)
        st["beta"] = BETA
        return st
    if kind == "scan":
        cells = st["cells"]
        st["rho"] = torch.cat([torch.from_numpy(w.rho.reshape(-1)) for w in cells]).to(DEV)
        st["solver"] = BatchSolver(cells, precision="mixed", workers=min(16, len(cells)), kgroups=1)
        st["lower"] = [6] * len(cells)
        return st
    form, tol = {"step": ("mixed", 1e-4), "fp64": ("fp64", 1e-11)}.get(kind, (case.get("form"), 0.0))
    bands = case["bands"] if kind != "apply" else _apply_bands((2 * case["M"] + 1) ** 3)
    st["solver"] = BandSolver(case["lattice"], _grid_of(case), case["M"], bands, wl.TUNGSTEN_CARBIDE, wl.EPOXY, st["Q"],
                              penal=PENAL, precision=form, tol=tol)
    if kind == "step":
        st["theta"].requires_grad_()
    if kind != "apply":
        st["weights"] = _weights(len(st["Q"]), bands)
    return st


# ---------------------------------------------------------------------------
# one pass

def run(st):
    kind = st["kind"]
    if kind == "map":
        dmap, opt = st["map"], st["opt"]
        rho = dmap.project(st["x"], st["beta"])
        gx = dmap.backprop(st["g"])
        # the third update of a run, from the two iterates before it and their asymptotes
        x = st["x"].clone()
        opt.xold1.copy_(st["x1"])
        opt.xold2.copy_(st["x2"])
        torch.sub(st["x1"], 0.5, out=opt.low)
        torch.add(st["x1"], 0.5, out=opt.upp)
        opt.iteration = 2
        opt.step(x, gx)
        return {"rho": rho, "gx": gx, "x": x, "low": opt.low, "upp": opt.upp}
    s = st["solver"]
    if kind == "scan":
        s.set_designs(st["rho"])
        om = s.bands()
        gaps, _ = s.gap_and_grad(n_lower=st["lower"], need_grad=False)
        return {"lambda": torch.cat([o.reshape(-1) for o in om]).square().float(), "gap": gaps.float()}
    if kind == "step":
        theta = st["theta"]
        theta.grad = None
        rho = torch.sigmoid(theta)
        s.set_design(rho)
        om = s.bands()
        val, g = s.gap_and_grad(mode=B.PC_GRAD_ALLBANDS, weights=st["weights"])
        rho.backward(g.to(rho.dtype))
        return {"lambda": om.square().to(rho.dtype), "value": val.to(rho.dtype), "grad": theta.grad}
    if kind == "fp64":
        s.set_design(st["rho"])
        om = s.bands()
        val, g = s.gap_and_grad(mode=B.PC_GRAD_ALLBANDS, weights=st["weights"])
        return {"lambda": om.square(), "value": val, "grad": g}
    s.set_design(st["rho"])
    ax, ox = s.apply_operator(0, st["x"])
    return {"ax": ax.to(st["x"].dtype), "ox": ox.to(st["x"].dtype)}


# ---------------------------------------------------------------------------
# what a pass cannot do without

def _setup_flops(n, M):
    """Separable structure factors of three fields and two Hermitian N x N inverses (complex)."""
    L, N = 4 * M + 1, (2 * M + 1) ** 3
    return 8.0 * 3 * (n[0] * n[1] * n[2] * L + n[0] * n[1] * L * L + n[0] * L ** 3) + 2 * 8.0 * N ** 3


def _solve_flops(n, M, nk, nb, grad):
    """One application of the operator pair and two Gram products per band, and the adjoint's
    synthesis of nine fields: the least a block method can check and differentiate nb bands with."""
    N, m2 = (2 * M + 1) ** 3, 2 * M + 1
    f = nk * (8.0 * 9 * N * N * nb + 2 * 8.0 * 3 * N * nb * nb)
    if grad:
        f += nk * nb * 8.0 * 9 * (m2 ** 3 * n[2] + m2 * m2 * n[1] * n[2] + m2 * n[0] * n[1] * n[2])
    return f


def work(case):
    kind = case["kind"]
    if kind == "map":
        n = _grid_of(case)
        ne = n[0] * n[1] * n[2]
        nv = ne // case["spacing"] ** 3 // (8 if case["octant"] else 1)
        return {"bytes": 8.0 * (2 * ne + 13 * nv), "flops": 30.0 * ne + 40.0 * nv}
    if kind == "scan":
        n = (case["n0"],) * 3
        ne, nd = case["n0"] ** 3, case["designs"]
        return {"bytes": nd * (8.0 * ne + 4.0 * case["nk"] * case["bands"]),
                "flops": nd * (_setup_flops(n, case["M"]) + _solve_flops(n, case["M"], case["nk"], case["bands"], False))}
    n, M = _grid_of(case), case["M"]
    ne, N = n[0] * n[1] * n[2], (2 * M + 1) ** 3
    if kind == "apply":
        return {"bytes": 8.0 * ne + 3 * (16.0 if case["form"] == "fp64" else 8.0) * 3 * N * case["cols"],
                "flops": _setup_flops(n, M) + 8.0 * 9 * N * N * case["cols"]}
    nk = case["nk"] if kind == "step" else len(_shifted_grid(case["grid"]))
    width = 4.0 if kind == "step" else 8.0
    return {"bytes": width * (2 * ne + nk * case["bands"]) + 8.0 * nk * case["bands"],
            "flops": _setup_flops(n, M) + _solve_flops(n, M, nk, case["bands"], True)}


# ---------------------------------------------------------------------------
# the same in 64 bits with plain torch

EXACT_MOST = 2.4e10  # wavevectors x (3N)^3 of dense eigenproblems that take a few seconds

def _lattice(lat):
    A = {"sc": np.eye(3),
         "bcc": 0.5 * np.array([[-1.0, 1, 1], [1, -1, 1], [1, 1, -1]]).T,
         "fcc": 0.5 * np.array([[0.0, 1, 1], [1, 0, 1], [1, 1, 0]]).T}[lat]
    return A, abs(np.linalg.det(A))


class _Cell:
    """Dense operators of one cell: T_rho and the two inverse compliance blocks, plane waves g in
    [-M, M]^3 (last index fastest), element sums at the voxel centroids."""

    def __init__(self, lat, rho, M, ph1, ph0, penal):
        self.n, self.M = tuple(rho.shape), M
        A, self.V = _lattice(lat)
        self.T = torch.tensor(np.linalg.inv(A).T, device=DEV)
        r = torch.arange(-M, M + 1, device=DEV)
        self.g = torch.stack(torch.meshgrid(r, r, r, indexing="ij"), -1).reshape(-1, 3)
        self.rho = rho.to(torch.float64)
        chi = self.rho ** penal
        self.dchi = penal * self.rho ** (penal - 1.0)
        f = lambda p: (p["rho"], (1 - 2 * p["nu"]) / p["E"], (1 + p["nu"]) / p["E"])  # noqa: E731
        self.d = [b - a for a, b in zip(f(ph0), f(ph1))]
        mats = [self._toeplitz(a + chi * d) for a, d in zip(f(ph0), self.d)]
        self.Tr, self.W = mats[0], [torch.linalg.inv(mats[1]), torch.linalg.inv(mats[2])]

    def _toeplitz(self, c):
        """V c^(g_q - g_p), c^(D) = mean of c exp(2 pi i D.s) over the centroids s."""
        w = [torch.exp(2j * math.pi * torch.arange(-2 * self.M, 2 * self.M + 1, device=DEV, dtype=torch.float64)[:, None]
                       * (torch.arange(k, device=DEV, dtype=torch.float64)[None] + 0.5) / k) for k in self.n]
        c = torch.einsum("ai,bj,cl,ijl->abc", w[0], w[1], w[2], c.to(torch.complex128)) / c.numel()
        d = self.g[None, :, :] - self.g[:, None, :] + 2 * self.M
        return self.V * c[d[..., 0], d[..., 1], d[..., 2]]

    def strain(self, Q):
        """B[s, c, p]: the plane waves' dilatational (s = 0) and five deviatoric strain components."""
        K = (torch.tensor(Q, device=DEV) + self.g.to(torch.float64)) @ self.T.T
        k0, k1, k2 = K.T
        z = torch.zeros_like(k0)
        r2, r3, r6 = 2 ** -0.5, 3 ** -0.5, 6 ** -0.5
        return torch.stack([torch.stack([k0 * r3, k1 * r3, k2 * r3]), torch.stack([k0 * r2, -k1 * r2, z]),
                            torch.stack([k0 * r6, k1 * r6, -2 * k2 * r6]), torch.stack([z, k2 * r2, k1 * r2]),
                            torch.stack([k2 * r2, z, k0 * r2]), torch.stack([k1 * r2, k0 * r2, z])])

    def apply(self, Q, x):
        """A x and Omega x, x (cols, 3N)."""
        N = self.g.shape[0]
        Bs, u = self.strain(Q), x.reshape(-1, 3, N)
        out = torch.zeros_like(u)
        for s in range(6):
            e = torch.einsum("cp,vcp->vp", Bs[s].to(u.dtype), u)
            out += Bs[s].to(u.dtype)[None] * (e @ self.W[min(s, 1)].T)[:, None, :]
        return ((2 * math.pi * self.V) ** 2 * out).reshape(x.shape), (u @ self.Tr.T).reshape(x.shape)

    def solve(self, Q, nb):
        """Lowest nb eigenvalues, eigenvectors (3, N, nb) and stress coefficients (6, N, nb)."""
        N = self.g.shape[0]
        Bs = self.strain(Q).to(torch.complex128)
        A = torch.zeros((3, N, 3, N), dtype=torch.complex128, device=DEV)
        for c in range(3):
            for d in range(3):
                for w in range(2):
                    part = Bs[:1] if w == 0 else Bs[1:]
                    A[c, :, d, :] += (part[:, c].T @ part[:, d]) * self.W[w]
        A = A.reshape(3 * N, 3 * N) * (2 * math.pi * self.V) ** 2
        Li = torch.linalg.inv(torch.linalg.cholesky(self.Tr))
        C = torch.einsum("pa,cadb,qb->cpdq", Li, A.reshape(3, N, 3, N), Li.conj()).reshape(3 * N, 3 * N)
        lam, y = torch.linalg.eigh((C + C.conj().T) / 2)
        theta = torch.einsum("ap,cav->cpv", Li.conj(), y[:, :nb].reshape(3, N, nb))
        e = torch.einsum("scp,cpv->spv", Bs, theta) * (2j * math.pi * self.V)
        sig = torch.stack([self.W[min(s, 1)] @ e[s] for s in range(6)])
        return lam[:nb], theta, sig

    def grad(self, weights, lam, theta, sig):
        """sum_b weights_b dlambda_b / drho_e on the voxel grid."""
        M2 = 2 * self.M + 1
        F = [torch.exp(2j * math.pi * (torch.arange(k, device=DEV, dtype=torch.float64)[:, None] + 0.5) / k
                       * torch.arange(-self.M, self.M + 1, device=DEV, dtype=torch.float64)[None]) for k in self.n]
        out = torch.zeros(self.n, dtype=torch.float64, device=DEV)
        for b in range(lam.numel()):
            f = torch.cat([theta[..., b], sig[..., b]]).reshape(9, M2, M2, M2)
            f = torch.einsum("cl,vijl->vijc", F[2], f)
            f = torch.einsum("bj,vijc->vibc", F[1], f)
            f = torch.einsum("ai,vibc->vabc", F[0], f)
            p = f.real ** 2 + f.imag ** 2
            out += float(weights[b]) * (-float(lam[b]) * self.d[0] * p[:3].sum(0) - self.d[1] * p[3] - self.d[2] * p[4:].sum(0))
        return out * self.dchi * self.V / out.numel()


def _evaluate(cell, Qs, nb, weights):
    lams, grad = [], torch.zeros(cell.n, dtype=torch.float64, device=DEV)
    for k, Q in enumerate(Qs):
        lam, theta, sig = cell.solve(Q, nb)
        lams.append(lam)
        if weights is not None:
            grad += cell.grad(weights[k].tolist(), lam, theta, sig)
    return torch.stack(lams), grad


def _map_exact(case, st):
    """The published formulas, node by node of the (small) neighbourhood of each voxel class."""
    n, sp = _grid_of(case), case["spacing"]
    A, _ = _lattice(case["lattice"])
    nd = [k // sp for k in n]
    x, beta = st["x"], BETA
    radius = 1.4 * np.linalg.norm(A[:, 0]) / n[0]
    if case["octant"]:
        idx = [torch.tensor([min(i, k - 1 - i) for i in range(k)], device=DEV) for k in nd]
        phi = x.reshape([k // 2 for k in nd])[idx[0]][:, idx[1]][:, :, idx[2]]
    else:
        phi = x.reshape(nd)
    mu = torch.empty(n, dtype=torch.float64, device=DEV)
    reach = range(-3, 4)
    offs = [(a, b, c) for a in reach for b in reach for c in reach]
    classes = [(a, b, c) for a in range(sp) for b in range(sp) for c in range(sp)]
    tables = []
    for p in classes:
        tab = []
        for o in offs:
            fr = [(sp * o[i] + 0.5 * sp - p[i] - 0.5) / n[i] for i in range(3)]
            w = radius - float(np.linalg.norm(A @ np.array(fr)))
            if w > 0:
                tab.append((o, w))
        tot = sum(w for _, w in tab)
        tables.append([(o, w / tot) for o, w in tab])
        acc = sum(w / tot * torch.roll(phi, [-o[0], -o[1], -o[2]], (0, 1, 2)) for o, w in tab)
        mu[p[0]::sp, p[1]::sp, p[2]::sp] = acc
    mu = mu.clamp(0, 1)
    em, eb = torch.exp(-beta * mu), math.exp(-beta)
    rho = (1 - em + mu * eb).clamp(0, 1)
    gm = st["g"] * (beta * em + eb)
    gphi = torch.zeros(nd, dtype=torch.float64, device=DEV)
    for p, tab in zip(classes, tables):
        gp = gm[p[0]::sp, p[1]::sp, p[2]::sp]
        for o, w in tab:
            gphi += w * torch.roll(gp, list(o), (0, 1, 2))
    if case["octant"]:
        h = [k // 2 for k in nd]
        gx = sum(t[:h[0], :h[1], :h[2]] for t in
                 [torch.flip(gphi, [ax for ax in range(3) if m >> ax & 1]) for m in range(8)])
    else:
        gx = gphi
    return rho, gx.reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    N = (2 * case.get("M", 1) + 1) ** 3
    st = _inputs(case, seed)
    if kind == "map":
        rho, gx = _map_exact(case, st)
        return {"rho": rho, "gx": gx, "x": None, "low": None, "upp": None}
    if kind == "scan":
        cells = st["cells"]
        if len(cells) * case["nk"] * (3 * N) ** 3 > EXACT_MOST:
            return None
        lam, gaps = [], []
        for w in cells:
            c = _Cell(w.lattice, torch.from_numpy(w.rho).to(DEV), w.M, w.phase1, w.phase0, 1.0)
            v = _evaluate(c, w.Q, w.nbands, None)[0].clamp(min=0)
            a, b = v[:, 5].max().sqrt(), v[:, 6].min().sqrt()
            lam.append(v.reshape(-1))
            gaps.append(2 * (b - a) / (b + a))
        return {"lambda": torch.cat(lam), "gap": torch.stack(gaps)}
    if kind == "apply":
        c = _Cell(case["lattice"], st["rho"], case["M"], wl.TUNGSTEN_CARBIDE, wl.EPOXY, PENAL)
        ax, ox = c.apply(st["Q"][0], st["x"].to(torch.complex128))
        return {"ax": ax, "ox": ox}
    Q = st["Q"]
    if len(Q) * (3 * N) ** 3 > EXACT_MOST:
        return None
    # the densities as run() makes them, widened
    rho = torch.sigmoid(st["theta"]).to(torch.float64) if kind == "step" else st["rho"]
    c = _Cell(case["lattice"], rho, case["M"], wl.TUNGSTEN_CARBIDE, wl.EPOXY, PENAL)
    w = _weights(len(Q), case["bands"])
    lam, g = _evaluate(c, Q, case["bands"], w)
    if kind == "step":
        g = g * rho * (1 - rho)
    return {"lambda": lam.clamp(min=0), "value": (w * lam).sum().reshape(1), "grad": g}
