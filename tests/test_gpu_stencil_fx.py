"""The real FP64 stencil works in fixed point with one scale per column: every FD order, grids
thinner than the stencil and around the tile width of 32, columns and potentials of any
magnitude, and non-finite values, against the oracle's H without projectors."""
import numpy as np
import pytest

from oracle import hubbard as o

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F64, Hub  # noqa: E402

EPS = 2.0 ** -53


def build(n, L, veff, n0):
    hb = Hub(n, L, n0, prec=HUB_F64)
    hb.set_veff(torch.tensor(veff, device="cuda"))
    hb.set_atoms([])
    return hb, o.Hamiltonian(o.Grid(n, L, (0, 0, 0), n0), veff, [])


def largest_sum(n, L, n0, veff):
    """Sum of |coefficients| of one row of H."""
    c0, c = o.fd_laplacian_weights(n0)
    kin = 0.5 * sum((n[a] / L[a]) ** 2 for a in range(3)) * (abs(c0) + 2 * np.sum(np.abs(c)))
    return kin + np.max(np.abs(veff))


def check(hb, ham, X, bound):
    Y = torch.empty(X.shape, dtype=torch.float64, device="cuda")
    with np.errstate(all="ignore"):
        ref = ham.apply(X.T).T
    for v in range(hb.get_tuning()["n_variants"]):
        hb.set_tuning(v)
        hb.apply_H(0, torch.tensor(X, device="cuda"), Y)
        got = Y.cpu().numpy()
        for j in range(X.shape[0]):
            fin = np.isfinite(ref[j])
            assert np.array_equal(fin, np.isfinite(got[j])), (v, j)
            top = np.max(np.abs(X[j][np.isfinite(X[j])]))
            # 40 roundings of partial sums on the oracle's side, the format's 2^-58 on the other
            assert np.max(np.abs(got[j] - ref[j])[fin], initial=0.0) <= 64 * EPS * bound * top, (v, j)


@pytest.mark.parametrize("n0", [1, 2, 3, 4, 5, 6])
def test_every_order(n0):
    rng = np.random.default_rng(n0)
    n, L = (14, 11, 9), (3.1, 2.7, 2.2)
    veff = rng.uniform(-5, 1, 14 * 11 * 9)
    hb, ham = build(n, L, veff, n0)
    check(hb, ham, rng.standard_normal((3, veff.size)), largest_sum(n, L, n0, veff))


@pytest.mark.parametrize("n", [(33, 9, 17), (32, 20, 5), (65, 3, 8), (1, 70, 2), (3, 150, 7), (31, 31, 1)])
def test_tile_edges(n):
    rng = np.random.default_rng(sum(n))
    L = tuple(0.21 * v for v in n)
    veff = rng.uniform(-5, 1, n[0] * n[1] * n[2])
    hb, ham = build(n, L, veff, 6)
    check(hb, ham, rng.standard_normal((2, veff.size)), largest_sum(n, L, 6, veff))


@pytest.mark.parametrize("vscale,hgrid", [(1.0, 0.2), (400.0, 0.2), (3e4, 0.2), (1e9, 0.2), (10.0, 2.0)])
def test_magnitudes(vscale, hgrid):
    """Columns from 1e-290 to 1e290 and zero (of their own scale each), potentials beyond the
    fixed-point range, a coarse grid."""
    rng = np.random.default_rng(5)
    n = (12, 13, 10)
    L = tuple(hgrid * v for v in n)
    veff = vscale * rng.uniform(-1, 1, n[0] * n[1] * n[2])
    hb, ham = build(n, L, veff, 6)
    X = rng.standard_normal((6, veff.size)) * np.array([1.0, 1e-290, 1e-30, 1e200, 1e290, 0.0])[:, None]
    X[0] *= np.exp(-30 * rng.random(veff.size))        # a wide range within the column
    check(hb, ham, X, largest_sum(n, L, 6, veff))


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_non_finite_stays_local(value):
    """One non-finite value reaches the points of its own stencil and nothing else."""
    rng = np.random.default_rng(6)
    n, L = (20, 21, 19), (4.0, 4.2, 3.8)
    veff = rng.uniform(-5, 1, n[0] * n[1] * n[2])
    hb, ham = build(n, L, veff, 6)
    X = rng.standard_normal((2, veff.size))
    X[1, 1234] = value
    check(hb, ham, X, largest_sum(n, L, 6, veff))


def test_filter_shift_and_aliasing():
    """The recurrence (alpha, beta, shift; Yprev aliasing Yout) against the oracle's filter."""
    rng = np.random.default_rng(8)
    n, L = (26, 18, 15), (5.2, 3.7, 3.1)
    veff = rng.uniform(-5, 1, n[0] * n[1] * n[2])
    hb, ham = build(n, L, veff, 6)
    X = rng.standard_normal((4, veff.size))
    b = largest_sum(n, L, 6, veff)
    ref = o.chebyshev_filter(ham, X.T, 9, 0.1 * b, b, -10.0).T
    Xd = torch.tensor(X, device="cuda")
    hb.chefsi_filter(0, Xd, 9, 0.1 * b, b, -10.0)
    # nine recurrence steps, each with the error of one application relative to its bound
    assert np.max(np.abs(Xd.cpu().numpy() - ref)) <= 9 * 9 * 64 * EPS * np.max(np.abs(X))
