"""The subspace eigensolver through hub_rayleigh_ritz: sizes around the groups of pairs the CTAs own
(none, one, several groups, odd sizes, a ragged last group), real and complex, random spectra and the
highly degenerate spectrum of the free-particle stencil on the whole space of a small grid, large
and small scales.

Bounds: the eigenvalues against numpy.linalg.eigh of the projected matrix; orthonormality and the
off-diagonal of the rotated projected matrix to 64 n ulp of the largest eigenvalue (a cyclic Jacobi
step costs a few ulp per element and sweep, the convergence threshold is 1e-13)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F64, Hub  # noqa: E402


def run(n, X0, v, cplx, scale):
    L = tuple(0.3 * m for m in n)
    dV = 0.3 ** 3
    hb = Hub(n, L, 6, prec=HUB_F64, complex_=cplx, kpt=(0.1, 0.2, -0.15) if cplx else None)
    hb.set_veff(torch.tensor(v * scale, device="cuda"))
    hb.set_atoms([])
    X = torch.tensor(X0, device="cuda").to(hb.dtype)
    Y = torch.empty_like(X)
    hb.apply_H(0, X, Y)
    H0 = dV * (X.conj() @ Y.T).cpu().numpy()
    eig = np.asarray(hb.rayleigh_ritz(0, X))
    hb.apply_H(0, X, Y)
    S = dV * (X.conj() @ X.T).cpu().numpy()
    Hs = dV * (X.conj() @ Y.T).cpu().numpy()
    ref = np.linalg.eigvalsh((H0 + H0.conj().T) / 2)
    top = max(np.max(np.abs(ref)), 1e-300)
    m = X.shape[0]
    tol = 64 * m * 2.0 ** -52 + 1e-12
    assert np.all(np.diff(eig) >= 0)
    assert np.max(np.abs(eig - ref)) <= tol * top
    assert np.max(np.abs(S - np.eye(m))) <= tol
    assert np.max(np.abs(Hs - np.diag(eig))) <= tol * top


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("ncol", [1, 2, 3, 11, 12, 13, 25, 58, 131, 348, 501])
def test_random_spectrum(ncol, cplx):
    rng = np.random.default_rng(ncol)
    n = (12, 10, 9)
    Nd = 1080
    A = rng.standard_normal((Nd, ncol)) + (1j * rng.standard_normal((Nd, ncol)) if cplx else 0)
    Q, _ = np.linalg.qr(A)
    v = rng.uniform(-50, 20, Nd)
    run(n, np.ascontiguousarray(Q.T) / 0.3 ** 1.5, v, cplx, 1.0)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("vscale", [0.0, 1e-30, 1e12])
def test_whole_space_of_a_small_grid(vscale, cplx):
    """V = 0: the plane waves of the grid, up to 48-fold degenerate; V huge: nearly diagonal."""
    n = (6, 6, 7)
    Nd = 252
    rng = np.random.default_rng(5)
    run(n, np.eye(Nd) / 0.3 ** 1.5, rng.uniform(-1, 1, Nd), cplx, vscale)
