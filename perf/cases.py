"""What is timed: the library's calls as an electronic-structure program makes them.

A case is one call (or the few calls that belong together) on one cell.  Cells are rutile-shaped
TiO2 supercells with displaced atoms (KB projectors s, p, d on every atom, a Hubbard d shell on
every Ti), spacings of 0.2 to 0.3 bohr, orbital counts of up to about 4.8 per atom, as in
workloads/synthetic.py.  Blocks are [orbital, grid point], x fastest.
"""
import math

import numpy as np
import torch

from paper_2507_23612_gb300 import HUB_F32, HUB_F64, HUB_MIXED_BF16, Hub, batch_filter, scf_params
from paper_2507_23612_gb300.binding import fermi_dirac

HARTREE_EV = 27.211386245988
LATTICE = (4.594 / 0.529177210903, 4.594 / 0.529177210903, 2.959 / 0.529177210903)
U = 0.305
TI = ((0.0, 0.0, 0.0), (0.5, 0.5, 0.5))
OX = ((U, U, 0.0), (1 - U, 1 - U, 0.0), (0.5 + U, 0.5 - U, 0.5), (0.5 - U, 0.5 + U, 0.5))
KB_L, KB_RS, KB_RC, HUB_RC = (0, 1, 2), (0.8, 0.8, 1.0), 2.5, 5.0
MP = ((0.25, 0.25, 0.25), (-0.25, 0.25, 0.25), (0.25, -0.25, 0.25), (0.25, 0.25, -0.25))
PREC = {"f64": HUB_F64, "f32": HUB_F32, "bf16": HUB_MIXED_BF16}


def _case(name, do, reps, n, ncol, prec="f64", bloch=False, degree=0, systems=1):
    c = {"do": do, "ra": reps[0], "rb": reps[1], "rc": reps[2], "n1": n[0], "n2": n[1], "n3": n[2],
         "ncol": ncol, "prec": prec, "bloch": bloch, "degree": degree, "systems": systems}
    return dict(c, name=name) if name else c


def listed():
    big, big_n = (2, 2, 3), (88, 88, 84)          # the 72-atom cell of the benchmark
    return [
        # one H application on a small block of a test-sized grid: the smallest call, launches count
        _case("apply-small-f64", "apply", (1, 1, 1), (24, 20, 28), 16),
        # the filter of the small cell (32 orbitals on about 24^3 points, degree 20)
        _case("filter-small-f64", "filter", (1, 1, 1), (24, 24, 24), 32, degree=20),
        # the filter of a 12-atom cell in float: every SCF of the warm-start family and of MD steps
        _case("filter-12-f32", "filter", (1, 1, 2), (44, 44, 56), 58, "f32", degree=24),
        # the filter of the 72-atom cell: the bulk of an SCF iteration, double and float
        _case("filter-72-f64", "filter", big, big_n, 348, degree=24),
        _case("filter-72-f32", "filter", big, big_n, 348, "f32", degree=24),
        # the filter at a Bloch wavevector, 48 atoms (the k-point SCF)
        _case("filter-48-bloch-f32", "filter", (2, 2, 2), (88, 88, 56), 230, "f32", True, 24),
        # four snapshot / k-point systems in one batched filter
        _case("batch-24-bloch-f32", "batch", (2, 2, 1), (88, 88, 28), 115, "f32", True, 24, 4),
        # Rayleigh-Ritz, occupations, D and density of the 72-atom block: the other half of an iteration
        _case("project-72-f64", "project", big, big_n, 348),
        _case("project-72-f32", "project", big, big_n, 348, "f32"),
        # Hubbard forces of the 72-atom block (once per MD step)
        _case("forces-72-f32", "forces", big, big_n, 348, "f32"),
        # the Hartree potential of the density SCF on the 72-atom grid
        _case("hartree-72", "hartree", big, big_n, 1),
        # a first SCF iteration of the 12-atom cell, two spins, through the SCF driver
        _case("scf-12-f64", "scf", (1, 1, 2), (44, 44, 56), 58, degree=8),
    ]


def draw(rng):
    while True:
        do = rng.choice(["apply", "filter", "filter", "filter", "project", "project", "forces", "batch", "hartree", "scf"])
        reps = (rng.randint(1, 2), rng.randint(1, 2), rng.randint(1, 3))
        h = rng.uniform(0.19, 0.33)
        # grids of any size, half of them multiples of 4 on every axis, as the generators make them
        n = tuple(max(12, round(LATTICE[a] * reps[a] / h) + rng.randint(-1, 1)) for a in range(3))
        if rng.random() < 0.5:
            n = tuple(4 * max(3, round(v / 4)) for v in n)
        atoms = 6 * reps[0] * reps[1] * reps[2]
        ncol = int(round(math.exp(rng.uniform(math.log(6), math.log(4.84 * atoms)))))
        prec = "f64" if do in ("hartree", "scf") else rng.choice(["f64", "f32"])
        if do == "project" and rng.random() < 0.25:
            prec = "bf16"
        bloch = do == "batch" or (do in ("apply", "filter") and rng.random() < 0.3)
        if do == "batch":
            prec = "f32"
        degree = {"filter": rng.randint(6, 24), "batch": rng.randint(6, 24), "scf": 8}.get(do, 0)
        systems = rng.randint(2, 4) if do == "batch" else 1
        c = _case(None, do, reps, n, 1 if do == "hartree" else ncol, prec, bloch, degree, systems)
        cost = n[0] * n[1] * n[2] * ncol * max(1, degree) * systems * (4 if bloch else 1)
        if do == "hartree" or cost <= 88 * 88 * 84 * 348 * 20:
            return c


# ------------------------------------------------------------------------------- inputs

class _Atom:
    pass


def _cell(c):
    n = (c["n1"], c["n2"], c["n3"])
    L = tuple(LATTICE[a] * (c["ra"], c["rb"], c["rc"])[a] for a in range(3))
    return n, L


def _system(c, seed):
    """Atoms (host), V_eff parameters and D of one displaced cell."""
    g = np.random.Generator(np.random.PCG64(seed))
    _, L = _cell(c)
    atoms = []
    for kind, frac in (("Ti", TI), ("O", OX)):
        for i in range(c["ra"]):
            for j in range(c["rb"]):
                for k in range(c["rc"]):
                    for f in frac:
                        a = _Atom()
                        a.ti = kind == "Ti"
                        a.pos = (np.array(f) + (i, j, k)) * np.array(LATTICE) + 0.1 * g.standard_normal(3)
                        a.kb_l, a.kb_rs, a.kb_rc = KB_L, KB_RS, KB_RC
                        a.kb_gamma = tuple(float(v) for v in g.uniform(0.5, 2.0, 3))
                        a.hub_l, a.hub_rs, a.hub_rc = (2 if a.ti else -1), 1.0, (HUB_RC if a.ti else 0.0)
                        a.hub_U = 3.5 / HARTREE_EV if a.ti else 0.0
                        atoms.append(a)
    nhub = sum(a.ti for a in atoms)
    A = g.uniform(-0.05, 0.05, (nhub, 5, 5))
    return atoms, 0.2 * np.eye(5)[None] + 0.5 * (A + A.transpose(0, 2, 1))


def _veff(c, atoms):
    """Periodic Gaussians: Ti -3 Ha of width 1.2 bohr, O -2 Ha of 0.9."""
    n, L = _cell(c)
    V = torch.zeros((n[2], n[1], n[0]), dtype=torch.float64, device="cuda")
    for a in atoms:
        A, w = (-3.0, 1.2) if a.ti else (-2.0, 0.9)
        ax = []
        for d in range(3):
            x = np.arange(n[d]) * (L[d] / n[d]) - a.pos[d]
            t = np.arange(-3, 4)[:, None] * L[d]
            ax.append(torch.tensor(np.exp(-(x - t) ** 2 / (2 * w * w)).sum(0), device="cuda"))
        V += A * ax[2][:, None, None] * ax[1][None, :, None] * ax[0][None, None, :]
    return V.reshape(-1)


def _kpt(c, i=0):
    _, L = _cell(c)
    return tuple(2 * math.pi * MP[i % 4][a] / L[a] for a in range(3)) if c["bloch"] else (0.0, 0.0, 0.0)


def _dtype(c):
    if c["prec"] == "f64":
        return torch.complex128 if c["bloch"] else torch.float64
    return torch.complex64 if c["bloch"] else torch.float32


def _noise(c, seed):
    """The starting orbitals of an SCF: normal deviates."""
    n, _ = _cell(c)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    real = torch.float64 if c["prec"] == "f64" else torch.float32
    X = torch.randn((c["ncol"], n[0] * n[1] * n[2] * (2 if c["bloch"] else 1)), generator=g, device="cuda", dtype=real)
    if c["bloch"]:
        X = torch.view_as_complex(X.reshape(c["ncol"], -1, 2)).mul_(math.sqrt(0.5))
    return X


def _smooth(c, seed):
    """Band-limited orbitals of falling weight, as a filtered block has them, of norm about one."""
    n, L = _cell(c)
    X = _noise(dict(c, bloch=False, prec="f32"), seed).reshape(c["ncol"], n[2], n[1], n[0])
    k2 = 0
    for d, ax in ((2, 0), (1, 1), (0, 2)):
        f = torch.fft.rfftfreq(n[d]) if d == 0 else torch.fft.fftfreq(n[d])
        k = f.to("cuda", torch.float64) * (2 * math.pi * n[d] / L[d])
        k2 = k2 + (k * k).reshape([-1 if a == ax else 1 for a in range(3)])
    damp = torch.exp(-k2 / (2 * 2.0 ** 2)).to(torch.float32)
    out = torch.empty(c["ncol"], n[0] * n[1] * n[2], dtype=_dtype(c), device="cuda")
    vol = L[0] * L[1] * L[2]
    for j in range(0, c["ncol"], 32):
        s = torch.fft.irfftn(torch.fft.rfftn(X[j:j + 32], dim=(1, 2, 3)) * damp, s=X.shape[1:], dim=(1, 2, 3))
        s = s.reshape(s.shape[0], -1)
        s = s / s.square().mean(1, keepdim=True).sqrt() / math.sqrt(vol)
        w = torch.logspace(0, -1, c["ncol"], device="cuda", dtype=torch.float32)[j:j + 32, None]
        out[j:j + 32] = (s * w).to(out.dtype)
    return out


def _bounds(c):
    """(a, b, a_low): the spectrum's ends from the stencil's largest symbol and the potential."""
    n, L = _cell(c)
    kin = 0.5 * sum(_symbol(n[d], L[d]).max().item() for d in range(3))
    lo, up = -8.0, kin + 12.0
    return lo + 0.1 * (up - lo), up, lo


def _hub(c, atoms, D, k=0, spins=1):
    n, L = _cell(c)
    hub = Hub(n, L, 6, kpt=_kpt(c, k), complex_=c["bloch"], prec=PREC[c["prec"]])
    hub.set_veff(_veff(c, atoms))
    hub.set_atoms(atoms)
    for s in range(spins):
        hub.set_occupation_matrix(s, D)
    return hub


def _occupations(c):
    """Falling occupations of a block whose eigenvalues are not asked for."""
    return np.linspace(1.0, 0.0, c["ncol"])


def _smearing(c):
    """(kT, electrons): double blocks at 0.005 Ha; float ones hot, as in their first iterations."""
    return (0.005 if c["prec"] == "f64" else 0.5), 2.0 * max(1, int(0.83 * c["ncol"]))


def _scf_params(c, n, natoms):
    return scf_params(nspin=2, ncol=c["ncol"], ld=n[0] * n[1] * n[2], degree=c["degree"], max_iter=100, first_passes=1,
                      lanczos_steps=10, pulay_history=7, natoms=natoms, pulay_beta=0.3, kT=0.05,
                      n_elec=float(2 * max(1, int(0.83 * c["ncol"]))), tol_e_atom=1e-7, tol_D=1e-4)


def _rho(c, seed):
    """A density of the cell: Gaussians on its atoms."""
    atoms, _ = _system(c, seed)
    return -_veff(c, atoms)


def prepare(case, seed):
    c, do = case, case["do"]
    n, _ = _cell(c)
    st = {"case": c, "degree": c["degree"]}
    atoms, D = _system(c, seed)
    if do == "batch":
        # two k-points of each snapshot
        st["hubs"], st["X0"] = [], []
        for i in range(c["systems"]):
            a_i, D_i = _system(c, seed + 7919 * (i // 2))
            st["hubs"].append(_hub(c, a_i, D_i, i))
            st["X0"].append(_noise(c, seed + 31 * i))
        st["X"] = [x.clone() for x in st["X0"]]
        st["bounds"] = [[v] * c["systems"] for v in _bounds(c)]
        return st
    st["hub"] = _hub(c, atoms, D, spins=2 if do == "scf" else 1)
    if do in ("apply", "filter"):
        st["X0"], st["X"] = _noise(c, seed), _noise(c, seed)
        st["bounds"] = _bounds(c)
    elif do in ("project", "forces"):
        st["X0"] = _smooth(c, seed)
        st["X"] = torch.empty_like(st["X0"])
        st["f"] = _occupations(c)
        st["smear"] = _smearing(c)
        if do == "project":
            st["rho"] = torch.empty(n[0] * n[1] * n[2], dtype=torch.float64, device="cuda")
    elif do == "hartree":
        st["rho"], st["V"] = _rho(c, seed), torch.empty(n[0] * n[1] * n[2], dtype=torch.float64, device="cuda")
    elif do == "scf":
        st["X0"] = [_smooth(c, seed + s) for s in range(2)]
        st["X"] = [torch.empty_like(x) for x in st["X0"]]
        st["v0"] = [_noise(dict(c, ncol=1), seed + 5 + s).reshape(-1) for s in range(2)]
        st["D0"] = np.stack([D, D])
        st["params"] = _scf_params(c, n, len(atoms))
    return st


# ------------------------------------------------------------------------------- the calls

def _narrow(c, v):
    """A result that a float handle reports in double: it has the precision of the handle."""
    v = torch.as_tensor(v)
    return v if c["prec"] == "f64" else v.to(torch.float32)


def run(st):
    c, do = st["case"], st["case"]["do"]
    if do == "apply":
        st["hub"].apply_H(0, st["X0"], st["X"])
        return st["X"]
    if do == "filter":           # works in place: a pass starts from the same block again
        st["X"].copy_(st["X0"])
        a, b, low = st["bounds"]
        st["hub"].chefsi_filter(0, st["X"], st["degree"], a, b, low)
        return st["X"]
    if do == "batch":
        for x, x0 in zip(st["X"], st["X0"]):
            x.copy_(x0)
        a, b, low = st["bounds"]
        batch_filter(st["hubs"], [0] * len(st["hubs"]), st["X"], st["degree"], a, b, low)
        return st["X"]
    if do == "project":
        hub, X = st["hub"], st["X"]
        X.copy_(st["X0"])
        eig = hub.rayleigh_ritz(0, X)
        kT, ne = st["smear"]
        f, _ = fermi_dirac(eig, 1.0, kT, ne, 2.0)
        D, _, eu = hub.occupation(0, X, f)
        st["rho"].zero_()
        hub.density(X, f, 2.0, st["rho"])
        # the orbitals themselves are fixed only up to sign and to rotations of degenerate ones
        return {"eig": _narrow(c, eig), "f": _narrow(c, f), "D": _narrow(c, D),
                "EU": _narrow(c, np.array([eu])), "rho": _narrow(c, st["rho"])}
    if do == "forces":
        return _narrow(c, st["hub"].hubbard_forces(0, st["X0"], st["f"]))
    if do == "hartree":
        st["V"].zero_()
        _, eh = st["hub"].hartree(st["rho"], st["V"], tol=1e-11)
        return {"V": st["V"], "EH": eh}
    if do == "scf":
        hub = st["hub"]
        for x, x0 in zip(st["X"], st["X0"]):
            x.copy_(x0)
        hub.scf_begin(st["params"], st["X"], st["v0"], st["D0"])
        r = hub.scf_iterate()
        eig, occ, D = hub.scf_get()
        return {"E": r["E"], "E_band": r["E_band"], "E_U": r["E_U"], "mu": r["mu"], "eig": eig, "occ": occ, "D": D}
    raise ValueError(do)


# ------------------------------------------------------------------------------- work

def work(case):
    c, do = case, case["do"]
    nd = c["n1"] * c["n2"] * c["n3"]
    real = 8 if c["prec"] == "f64" else 4
    block = nd * c["ncol"] * real * (2 if c["bloch"] else 1)
    cells = c["ra"] * c["rb"] * c["rc"]
    h3 = LATTICE[0] * LATTICE[1] * LATTICE[2] * cells / nd
    sphere = lambda r: 4 / 3 * math.pi * r ** 3 / h3                     # noqa: E731
    funcs = cells * (6 * 9 * sphere(KB_RC) + 2 * 5 * sphere(HUB_RC))     # function-points of the projectors
    # 44 flops per point for the Laplacian, V and the recurrence, 4 per function-point and orbital
    h_flops = c["ncol"] * (44 * nd + 4 * funcs) * (3 if c["bloch"] else 1)
    if do == "apply":
        return {"bytes": 2 * block, "flops": h_flops}
    if do in ("filter", "batch"):
        # the block in and out, and per degree the block, its predecessor and the result
        return {"bytes": c["systems"] * 3 * block * c["degree"], "flops": c["systems"] * h_flops * c["degree"]}
    if do == "project":
        return {"bytes": 6 * block, "flops": h_flops + 2.0 * nd * c["ncol"] ** 2 * 2}
    if do == "forces":
        return {"bytes": block, "flops": c["ncol"] * (3 * 24 * nd + 4 * 2 * cells * 10 * sphere(HUB_RC))}
    if do == "hartree":
        return {"bytes": 3 * 8 * nd, "flops": 300 * 50 * nd}
    return {"bytes": 2 * block * (3 * c["degree"] + 6), "flops": 2 * (h_flops * (c["degree"] + 11) + 4.0 * nd * c["ncol"] ** 2)}


# ------------------------------------------------------------------------------- 64-bit values

def _fact(k):
    return math.factorial(k)


def _lap_weights():
    c = [2.0 * (-1) ** (p + 1) * _fact(6) ** 2 / (p * p * _fact(6 - p) * _fact(6 + p)) for p in range(1, 7)]
    return -2.0 * sum(1.0 / (p * p) for p in range(1, 7)), c


def _symbol(n, L):
    """Minus the 1-D Laplacian's symbol on the n wavenumbers of a periodic line."""
    c0, c = _lap_weights()
    t = torch.arange(n, dtype=torch.float64) * (2 * math.pi / n)
    s = c0 + sum(2 * c[p - 1] * torch.cos(p * t) for p in range(1, 7))
    return -s * (n / L) ** 2


class _Exact:
    """The Hamiltonian in 64 bits, from its definition."""

    def __init__(self, c, atoms, D, k=0):
        self.c, (self.n, self.L) = c, _cell(c)
        self.kpt = _kpt(c, k)
        self.dV = np.prod([self.L[a] / self.n[a] for a in range(3)])
        self.V = _veff(c, atoms)
        self.sites = []
        ih = 0
        for a in atoms:
            gam = np.concatenate([[g] * (2 * l + 1) for l, g in zip(KB_L, a.kb_gamma)])
            self.sites.append((*self._table(a.pos, list(zip(KB_L, KB_RS)), KB_RC), torch.tensor(np.diag(gam), device="cuda"), False))
            if a.ti:
                M = 0.5 * a.hub_U * (np.eye(5) - 2.0 * D[ih])
                self.sites.append((*self._table(a.pos, [(2, 1.0)], HUB_RC), torch.tensor(M, device="cuda"), True))
                ih += 1

    def _table(self, R, channels, rc):
        """(grid index, value) pairs of every image, the functions along the last axis."""
        ax = []
        for d in range(3):
            h = self.L[d] / self.n[d]
            lo, hi = math.ceil((R[d] - rc) / h), math.floor((R[d] + rc) / h)
            ax.append(torch.arange(lo, hi + 1, device="cuda"))
        i = torch.meshgrid(*ax, indexing="ij")
        d = [i[a].double() * (self.L[a] / self.n[a]) - R[a] for a in range(3)]
        r2 = d[0] ** 2 + d[1] ** 2 + d[2] ** 2
        sel = r2 < rc * rc
        x, y, z, r2 = (v[sel] for v in (*d, r2))
        idx, angle = 0, 0.0
        for a in (2, 1, 0):
            ia = i[a][sel]
            idx = idx * self.n[a] + torch.remainder(ia, self.n[a])
            # an image in the cell number w on: node ia belongs to the atom's image at -w cells
            angle = angle - self.kpt[a] * self.L[a] * torch.div(ia, self.n[a], rounding_mode="floor").double()
        cols = []
        for l, rs in channels:
            N = math.sqrt(2.0 / (math.gamma(l + 1.5) * rs ** (2 * l + 3)))
            g = N * torch.exp(-r2 / (2 * rs * rs))
            if l == 0:
                Y = [0.5 / math.sqrt(math.pi) * torch.ones_like(x)]
            elif l == 1:
                k = math.sqrt(3 / (4 * math.pi))
                Y = [k * y, k * z, k * x]
            else:
                k1, k0, k2 = 0.5 * math.sqrt(15 / math.pi), 0.25 * math.sqrt(5 / math.pi), 0.25 * math.sqrt(15 / math.pi)
                Y = [k1 * x * y, k1 * y * z, k0 * (2 * z * z - x * x - y * y), k1 * x * z, k2 * (x * x - y * y)]
            cols += [g * v for v in Y]
        vals = torch.stack(cols, 1)
        if self.c["bloch"]:
            vals = vals * torch.polar(torch.ones_like(angle), angle)[:, None]
        return idx, vals

    def _axis(self, X, a, weights, sign, centre):
        """sum_p w_p (x_{+p} + sign x_{-p}) along axis a with the Bloch wrap, plus centre x."""
        v = X.reshape(X.shape[0], self.n[2], self.n[1], self.n[0])
        dim, n = 3 - a, self.n[a]
        out = centre * v if centre else torch.zeros_like(v)
        for p, w in enumerate(weights, 1):
            for s, f in ((p, 1.0), (-p, sign)):
                sh = torch.roll(v, -s, dim)
                if self.c["bloch"]:
                    j = torch.arange(n, dtype=torch.float64, device="cuda") + s
                    ph = self.kpt[a] * self.L[a] * torch.floor(j / n)
                    sh = sh * torch.polar(torch.ones_like(ph), ph).reshape([-1 if d == dim else 1 for d in range(4)])
                out += (f * w) * sh
        return out.reshape(X.shape)

    def apply(self, X):
        c0, w = _lap_weights()
        Y = torch.empty_like(X)
        for j in range(0, X.shape[0], 64):
            x = X[j:j + 64]
            y = self.V * x
            for a in range(3):
                q = -0.5 * (self.n[a] / self.L[a]) ** 2
                y += self._axis(x, a, [q * v for v in w], 1.0, q * c0)
            Y[j:j + 64] = y
        for idx, vals, M, _ in self.sites:
            C = self.dV * (X[:, idx] @ vals.conj())
            Y.index_add_(1, idx, (C @ M.to(C.dtype).T) @ vals.T)
        return Y

    def filter(self, X, m, a, b, low):
        e, c = 0.5 * (b - a), 0.5 * (b + a)
        s = e / (low - c)
        tau = 2.0 / s
        Y = (self.apply(X) - c * X) * (s / e)
        for _ in range(2, m + 1):
            sn = 1.0 / (tau - s)
            Y, X, s = (self.apply(Y) - c * Y) * (2 * sn / e) - (s * sn) * X, Y, sn
        return Y

    def ritz(self, X):
        S = self.dV * (X @ X.T)
        H = self.dV * (X @ self.apply(X).T)
        Li = torch.linalg.inv(torch.linalg.cholesky(S.cpu()))
        H = Li @ (0.5 * (H + H.T)).cpu() @ Li.T
        lam, Q = torch.linalg.eigh(0.5 * (H + H.T))
        return lam, (Q.T @ Li).cuda() @ X

    def project(self, X, f):
        """D of every Hubbard atom and E_U."""
        f = torch.as_tensor(f, device="cuda", dtype=torch.float64)
        D = []
        for idx, vals, _, hub in self.sites:
            if hub:
                C = self.dV * (X[:, idx] @ vals)
                D.append(C.T @ (f[:, None] * C))
        D = torch.stack(D)
        eu = 0.5 * 3.5 / HARTREE_EV * (D.diagonal(dim1=1, dim2=2).sum() - (D * D).sum())
        return D, eu

    def forces(self, X, f, D):
        f = torch.as_tensor(f, device="cuda", dtype=torch.float64)
        w = [(-1) ** (p + 1) * _fact(6) ** 2 / (p * _fact(6 - p) * _fact(6 + p)) for p in range(1, 7)]
        hubs = [s for s in self.sites if s[3]]
        F = torch.zeros(len(hubs), 3, dtype=torch.float64)
        for a in range(3):
            G = torch.cat([self._axis(X[j:j + 64], a, [v * self.n[a] / self.L[a] for v in w], -1.0, 0.0)
                           for j in range(0, X.shape[0], 64)])
            for i, (idx, vals, M, _) in enumerate(hubs):
                C, g = self.dV * (X[:, idx] @ vals), self.dV * (G[:, idx] @ vals)
                F[i, a] = -2.0 * torch.sum(f[:, None] * g * (C @ M.T)).cpu()
        return F


def _fermi(e, kT, ne, deg):
    e = np.asarray(e)
    lo, hi = e.min() - 50 * kT, e.max() + 50 * kT
    for _ in range(200):
        mu = 0.5 * (lo + hi)
        s = np.sum(deg * 0.5 * (1 - np.tanh((e - mu) / (2 * kT))))
        lo, hi = (mu, hi) if s < ne else (lo, mu)
    mu = 0.5 * (lo + hi)
    return 0.5 * (1 - np.tanh((e - mu) / (2 * kT))), mu


def exact(case, seed):
    c, do = case, case["do"]
    wide = torch.complex128 if c["bloch"] else torch.float64
    if do == "batch":
        out = []
        for i in range(c["systems"]):
            a_i, D_i = _system(c, seed + 7919 * (i // 2))
            out.append(_Exact(c, a_i, D_i, i).filter(_noise(c, seed + 31 * i).to(wide), c["degree"], *_bounds(c)))
        return out
    atoms, D = _system(c, seed)
    n, L = _cell(c)
    if do == "hartree":
        rho = _rho(c, seed).reshape(n[2], n[1], n[0])
        sym = sum(_symbol(n[d], L[d]).reshape([-1 if a == 2 - d else 1 for a in range(3)]) for d in range(3)).cuda()
        sym[0, 0, 0] = 1.0
        R = 4 * math.pi * torch.fft.fftn(rho) / sym
        R[0, 0, 0] = 0.0
        V = torch.fft.ifftn(R).real.reshape(-1)
        dV = L[0] * L[1] * L[2] / V.numel()
        return {"V": V, "EH": float(0.5 * dV * torch.dot(rho.reshape(-1), V))}
    H = _Exact(c, atoms, D)
    if do == "apply":
        return H.apply(_noise(c, seed).to(wide))
    if do == "filter":
        return H.filter(_noise(c, seed).to(wide), c["degree"], *_bounds(c))
    if do == "project":
        lam, X = H.ritz(_smooth(c, seed).double())
        kT, ne = _smearing(c)
        f, _ = _fermi(lam.numpy(), kT, ne, 2.0)
        Db, eu = H.project(X, f)
        rho = 2.0 * (torch.as_tensor(f, device="cuda")[:, None] * X * X).sum(0)
        return {"eig": lam, "f": f, "D": Db, "EU": np.array([eu.item()]), "rho": rho}
    if do == "forces":
        F = torch.zeros(len(atoms), 3, dtype=torch.float64)
        F[[i for i, a in enumerate(atoms) if a.ti]] = H.forces(_smooth(c, seed).double(), _occupations(c), D)
        return F
    # scf: Lanczos bounds, one filter and Rayleigh-Ritz per spin, Fermi level, D, energies
    p = _scf_params(c, n, len(atoms))
    eig, Xs = [], []
    for s in range(2):
        v = _noise(dict(c, ncol=1), seed + 5 + s)
        v, last, beta, al, be = v / v.norm(), torch.zeros_like(v), 0.0, [], []
        for _ in range(10):
            w = H.apply(v) - beta * last
            al.append(float((v * w).sum()))
            w = w - al[-1] * v
            beta = float(w.norm())
            be.append(beta)
            last, v = v, w / beta
        r = np.linalg.eigvalsh(np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1))
        lo, up = r[0], r[-1] + be[-1]
        lam, X = H.ritz(H.filter(_smooth(c, seed + s), c["degree"], lo + 0.1 * (up - lo), up, lo))
        eig.append(lam.numpy())
        Xs.append(X)
    eig = np.stack(eig)
    f, mu = _fermi(eig, p.kT, p.n_elec, 1.0)
    Ds, eu = zip(*(H.project(Xs[s], f[s]) for s in range(2)))
    Ds, eu = torch.stack(Ds), float(sum(eu))
    M = torch.tensor(0.5 * 3.5 / HARTREE_EV * (np.eye(5) - 2.0 * D), device="cuda")
    g = np.clip(f, 1e-300, 1 - 1e-16)
    entropy = -float(np.sum(g * np.log(g) + (1 - g) * np.log(1 - g)))
    band = float(np.sum(f * eig))
    return {"E": band - float((M * Ds).sum()) + eu - p.kT * entropy, "E_band": band, "E_U": eu, "mu": float(mu),
            "eig": eig, "occ": f, "D": Ds}
