"""Localized columns: where a column is far below its maximum, H x and the projector products keep the
accuracy of their neighbourhood.  Columns decay along x by 1e-24 (1e-9 in float) to the far end of the
cell; errors are bounded against the largest |x| within 70 points along x (a tile of 32 points with a
halo of 6, and the pieces of 32 points that it meets)."""
import numpy as np
import pytest

from oracle import hubbard as o

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F32, HUB_F64, Hub  # noqa: E402

N, H = (512, 16, 12), 0.25
L = tuple(H * m for m in N)
ND = N[0] * N[1] * N[2]


def localized(ncol, cplx, decay):
    """Random signs and magnitudes times decay^(d / 256), d the distance along x from a centre of its own."""
    rng = np.random.default_rng(ncol)
    d = np.abs(np.arange(N[0])[None] - rng.integers(0, N[0], ncol)[:, None])
    env = decay ** (np.minimum(d, N[0] - d) / 256.0)
    X = rng.uniform(0.5, 1.0, (ncol, N[2] * N[1], N[0])) * rng.choice([-1.0, 1.0], (ncol, N[2] * N[1], N[0])) * env[:, None]
    X = X.reshape(ncol, ND)
    return X * np.exp(1j * rng.uniform(0, 6.28, (ncol, ND))) if cplx else X


def nearby(X, reach=70):
    """Largest |x| within `reach` points along x, of every (column, point)."""
    top = np.max(np.abs(X).reshape(X.shape[0], -1, N[0]), axis=1)
    return np.max([np.roll(top, s, axis=1) for s in range(-reach, reach + 1)], axis=0)


class _Atom:
    def __init__(self, pos):
        self.pos, self.kb_l, self.kb_rs, self.kb_gamma, self.kb_rc = np.asarray(pos), (0, 1, 2), (0.8, 0.8, 1.0), (0.7, 1.1, 0.9), 3.5
        self.hub_l, self.hub_rs, self.hub_rc, self.hub_U = -1, 1.0, 0.0, 0.0


def atoms():
    return [_Atom((L[0] * (i + 0.37) / 24, L[1] * ((7 * i) % 24 + 0.2) / 24, L[2] * ((5 * i) % 24 + 0.6) / 24)) for i in range(24)]


def tables(ats, kpt):
    g = o.Grid(N, L, kpt)
    cols = []
    for a in ats:
        idx, v = o.atom_function_table(g, a.pos, list(zip(a.kb_l, a.kb_rs)), a.kb_rc)
        B = np.zeros((ND, v.shape[1]), dtype=v.dtype)
        B[idx] = v
        cols.append(B)
    return g, np.concatenate(cols, axis=1)


def test_stencil():
    """H = -1/2 Lap + V of real doubles: elements are off by 2^-59 of the largest nearby, the result by
    that times the row sum, with as much again for its own roundings."""
    rng = np.random.default_rng(1)
    veff = rng.uniform(-3, 1, ND)
    hb = Hub(N, L, 6, prec=HUB_F64)
    hb.set_veff(torch.tensor(veff, device="cuda"))
    hb.set_atoms([])
    X = localized(5, False, 1e-24)
    ref = o.Hamiltonian(o.Grid(N, L), veff, []).apply(X.T).T
    c0, c = o.fd_laplacian_weights(6)
    row = 1.5 / H ** 2 * (abs(c0) + 2 * np.sum(np.abs(c))) + 3.0
    bound = 2.0 ** -58 * row * nearby(X)[:, None] + 64 * 2.0 ** -53 * row * nearby(X, 6)[:, None]
    Y = torch.empty(X.shape, dtype=torch.float64, device="cuda")
    for v in range(hb.get_tuning()["n_variants"]):
        hb.set_tuning(v)
        hb.apply_H(0, torch.tensor(X, device="cuda"), Y)
        err = np.abs(Y.cpu().numpy() - ref).reshape(5, -1, N[0])
        assert np.all(err <= bound), v


@pytest.mark.parametrize("prec,cplx", [(HUB_F64, False), (HUB_F64, True), (HUB_F32, True)])
def test_gather(prec, cplx):
    kpt = (0.05, 0.2, -0.3) if cplx else (0.0, 0.0, 0.0)
    ats = atoms()
    g, P = tables(ats, kpt)
    hb = Hub(N, L, 6, prec=prec, complex_=cplx, kpt=kpt if cplx else None)
    hb.set_atoms(ats if prec == HUB_F64 else ats * 4)   # (as many as the digit form takes in float)
    X = localized(130, cplx, 1e-24 if prec == HUB_F64 else 1e-9)
    X = torch.tensor(X, device="cuda").to(hb.dtype)
    hb.profile(1)
    C = hb.project(X)[:P.shape[1]]
    assert "copy" in hb.profile_read()                  # the digit form ran
    hb.profile(-1)
    X = X.cpu().numpy().astype(np.complex128 if cplx else np.float64)
    ref = g.dV * (P.conj().T @ X.T)
    # 16 u per point of the support, of the largest |x| near it and the function's largest value
    u = 2.0 ** -53 if prec == HUB_F64 else 2.0 ** -24
    near = nearby(X, 40)
    inside = (np.abs(P) > 0).reshape(-1, N[0], P.shape[1]).any(0)            # x planes of every function
    top = np.array([np.max(near[:, inside[:, p]], axis=1) for p in range(P.shape[1])])
    pts = np.count_nonzero(P, axis=0)[:, None]
    assert np.all(np.abs(C - ref) <= 16 * u * g.dV * top * np.max(np.abs(P), axis=0)[:, None] * pts)


@pytest.mark.parametrize("prec,cplx", [(HUB_F64, False), (HUB_F64, True), (HUB_F32, True)])
def test_scatter(prec, cplx):
    """Coefficients that decay with the atoms' distance from a centre of each column."""
    kpt = (0.05, 0.2, -0.3) if cplx else (0.0, 0.0, 0.0)
    ats = atoms()
    g, P = tables(ats, kpt)
    hb = Hub(N, L, 6, prec=prec, complex_=cplx, kpt=kpt if cplx else None)
    copies = 1 if prec == HUB_F64 else 4
    hb.set_atoms(ats * copies)
    rng = np.random.default_rng(3)
    ncol = 130
    x = np.repeat([a.pos[0] / L[0] for a in ats], 9)
    d = np.abs(x[:, None] - rng.uniform(0, 1, ncol)[None])
    W = rng.uniform(0.5, 1.0, (P.shape[1], ncol)) * (1e-24 if prec == HUB_F64 else 1e-9) ** (2 * np.minimum(d, 1 - d))
    W = W * np.exp(1j * rng.uniform(0, 6.28, W.shape)) if cplx else W
    Y = torch.zeros(ncol, ND, dtype=hb.dtype, device="cuda")
    hb.profile(1)
    hb.expand(np.concatenate([W] * copies), Y, 1.0)
    assert hb.profile_read()["scatter"][1] == 2             # maxima of W, then the digit form
    hb.profile(-1)
    got = Y.cpu().numpy().reshape(ncol, -1, N[0])
    W = W.astype({HUB_F64: np.complex128, HUB_F32: np.complex64}[prec]) if cplx else W
    ref = copies * (P @ W).T.reshape(ncol, -1, N[0])
    # of the coefficients of functions on the same brick: those whose x planes come within 8 points
    inside = (np.abs(P) > 0).reshape(-1, N[0], P.shape[1]).any(0)
    inside = np.any([np.roll(inside, s, axis=0) for s in range(-8, 9)], axis=0)
    top = np.array([np.max(np.abs(W) * inside[i][:, None], axis=0) for i in range(N[0])]).T
    u = 2.0 ** -53 if prec == HUB_F64 else 2.0 ** -24
    terms = copies * np.count_nonzero(inside, axis=1)
    assert np.all(np.abs(got - ref) <= (16 * u * np.max(np.abs(P)) * terms * top)[:, None])


@pytest.mark.parametrize("prec,ncol", [(HUB_F64, 12), (HUB_F64, 70), (HUB_F32, 140)])
def test_rotation(prec, ncol):
    """Orbitals with a common tail (a molecule and its vacuum): Rayleigh-Ritz returns X Q, and the rows of
    the tail follow the Q that the rows of the molecule give, to rounding of their own size times the
    condition of that fit (below 100)."""
    n = (512, 16, 10)
    Nd = n[0] * n[1] * n[2]
    rng = np.random.default_rng(5)
    d = np.abs(np.arange(512) - 256)
    env = (1e-24 if prec == HUB_F64 else 1e-9) ** (d / 256.0)
    hb = Hub(n, tuple(H * m for m in n), 6, prec=prec)
    hb.set_veff(torch.tensor(rng.uniform(-1, 0, Nd), device="cuda"))
    hb.set_atoms([])
    X = torch.tensor((rng.standard_normal((ncol, n[1] * n[2], 512)) * env).reshape(ncol, Nd), device="cuda").to(hb.dtype)
    X0 = X.double().cpu().numpy().reshape(ncol, -1, 512)
    hb.rayleigh_ritz(0, X)
    Y = X.double().cpu().numpy().reshape(ncol, -1, 512)
    core = slice(236, 276)
    Q = np.linalg.lstsq(X0[:, :, core].reshape(ncol, -1).T, Y[:, :, core].reshape(ncol, -1).T, rcond=None)[0]
    err = np.abs(Y - np.einsum("kj,kyx->jyx", Q, X0)).max(axis=(0, 1))
    size = np.abs(X0).max(axis=(0, 1)) * np.abs(Q).sum(axis=0).max()
    u = 2.0 ** -53 if prec == HUB_F64 else 2.0 ** -24
    assert np.all(err <= 100 * 16 * u * size)
