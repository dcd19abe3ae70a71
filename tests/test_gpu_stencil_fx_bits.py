"""How many bits the fixed-point stencil keeps: elements are rounded to nearest (2^-59 of the column's
maximum), and the Laplacian's factors keep theirs on grids of any spacing.  Alternating signs add
every point's error up: H x = lambda x with lambda the largest kinetic energy."""
import math
from fractions import Fraction

import numpy as np
import pytest

from oracle import hubbard as o

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F64, Hub  # noqa: E402


def alternating(n):
    i, j, k = np.meshgrid(np.arange(n[0]), np.arange(n[1]), np.arange(n[2]), indexing="ij")
    return np.where((i + j + k) % 2 == 0, 1.0, -1.0).transpose(2, 1, 0).reshape(-1)


def largest_kinetic(n, L):
    _, c = o.fd_laplacian_weights(6)
    c = np.asarray(c, dtype=np.longdouble)
    c0 = -2 * np.sum(c)
    one = np.longdouble(0.5) * (-c0 + 2 * np.sum(np.abs(c)))
    return sum((np.longdouble(n[a]) / np.longdouble(L[a])) ** 2 * one for a in range(3))


def apply(n, L, veff, x):
    hb = Hub(n, L, 6, prec=HUB_F64)
    hb.set_veff(torch.tensor(veff, device="cuda"))
    hb.set_atoms([])
    out = []
    for v in range(hb.get_tuning()["n_variants"]):
        hb.set_tuning(v)
        y = torch.empty((1, x.size), dtype=torch.float64, device="cuda")
        hb.apply_H(0, torch.tensor(x[None], device="cuda"), y)
        out.append(y.cpu().numpy()[0])
    return out


def test_elements_are_rounded_to_nearest():
    """One element of 1 sets the scale (units of 2^-58); all others are k + 0.95 units.  Rounded, each
    is off by 0.05 units and never by more than 0.5: lambda 2^-59 in the sum, the rounding of the
    sum to its own unit included (0.5 of lambda 2^-59 at this spacing).  Cut off, lambda 0.95 2^-58."""
    n = (32, 28, 26)
    h = 0.20366                              # the Laplacian's factor just below a power of two
    L = tuple(h * v for v in n)
    rng = np.random.default_rng(2)
    x = alternating(n) * (rng.integers(1, 1000) + 0.95) * 2.0 ** -58
    exact = x * float(largest_kinetic(n, L))
    spike = np.zeros(n[::-1], dtype=bool)
    spike[:, :, :7] = spike[:, :7, :] = spike[:7, :, :] = True          # what the point at the corner reaches
    spike[:, :, -7:] = spike[:, -7:, :] = spike[-7:, :, :] = True
    x[0] = 1.0
    for y in apply(n, L, np.zeros(x.size), x):
        assert np.max(np.abs(y - exact)[~spike.reshape(-1)]) <= float(largest_kinetic(n, L)) * 2.0 ** -59


@pytest.mark.parametrize("h", [(0.3, 0.31, 0.29), (1.0, 1.1, 1.3), (2.3, 2.0, 2.7), (4.1, 4.5, 4.9), (10.3, 11.9, 13.7),
                               (16.3, 12.9, 14.1), (31.0, 28.0, 90.0)])
@pytest.mark.parametrize("v", [0.0, 0.9])
def test_factors_keep_their_bits(h, v):
    """Two roundings at 2^-53 of the sum: the factors and V (2^-54 and 2^-55 of it or less) with the
    conversion of the result (2^-53).  V = 0.9 at one point, where x is zero."""
    n = (12, 14, 10)
    L = tuple(h[a] * n[a] for a in range(3))
    x = alternating(n)
    veff = np.zeros(x.size)
    far = np.ones(x.size, dtype=bool)
    if v:
        veff[0] = v
        x[0] = 0.0
        g = np.zeros(n[::-1], dtype=bool)
        g[0, 0, :] = g[0, :, 0] = g[:, 0, 0] = True                     # points on an axis through the zero
        far = ~g.reshape(-1)
    lam = float(largest_kinetic(n, L))
    for y in apply(n, L, veff, x):
        assert np.max(np.abs(y - lam * x)[far]) <= 2 * 2.0 ** -53 * lam + 2.0 ** -53 * lam      # and lambda itself


@pytest.mark.parametrize("h", [0.3, 1.0, 4.1, 12.9])
def test_potential_keeps_its_bits(h):
    """x = 1 everywhere: H x = V.  Bound: one rounding at 2^-53 of the row sum, as the FP64 sum has."""
    n = (12, 14, 10)
    L = tuple(h * m for m in n)
    x = np.ones(n[0] * n[1] * n[2])
    veff = np.random.default_rng(3).uniform(-0.9, 0.9, x.size)
    lam = float(largest_kinetic(n, L))
    for y in apply(n, L, veff, x):
        assert np.all(np.abs(y - veff) <= 2.0 ** -53 * (lam + np.abs(veff)))


@pytest.mark.parametrize("h", [0.3, 1.0, 4.1, 12.9])
def test_products_with_the_potential_keep_their_bits(h):
    """x = 1/3 everywhere, whose low limb is not zero: H x = V / 3, to one rounding at 2^-53 of the row sum."""
    n = (12, 14, 10)
    L = tuple(h * m for m in n)
    x = np.full(n[0] * n[1] * n[2], 1.0 / 3.0)
    veff = np.random.default_rng(4).uniform(-0.9, 0.9, x.size)
    lam = float(largest_kinetic(n, L))
    for y in apply(n, L, veff, x):
        assert np.all(np.abs(y - veff * x) <= 2.0 ** -53 * (lam + np.abs(veff)) * x)


@pytest.mark.parametrize("h", [(0.36, 0.36, 0.36), (0.1973, 0.1973, 0.1973), (0.6, 0.7, 0.8)])
def test_factors_do_not_shift_the_kinetic_energy(h):
    """256 amplitudes of the alternating column: the roundings of the results average to 2^-58 of lambda
    (2^-54.3 / 16), an error of the factors stays: at most 2^-55 together.  (The sum of the weights of
    order 12 that alternate, 4 sum over odd p, exactly.)"""
    n = (12, 14, 10)
    L = tuple(h[a] * n[a] for a in range(3))
    hb = Hub(n, L, 6, prec=HUB_F64)
    hb.set_veff(torch.zeros(12 * 14 * 10, dtype=torch.float64, device="cuda"))
    hb.set_atoms([])
    amp = np.random.default_rng(6).uniform(1.0, 2.0, 256)
    X = torch.tensor(amp[:, None] * alternating(n)[None], device="cuda")
    Y = torch.empty_like(X)
    hb.apply_H(0, X, Y)
    x, y = X.cpu().numpy().astype(np.longdouble), Y.cpu().numpy().astype(np.longdouble)
    f = math.factorial
    odd = sum(Fraction(2 * f(6) ** 2, p * p * f(6 - p) * f(6 + p)) for p in (1, 3, 5))
    lam = sum(np.longdouble(2) * np.longdouble(odd.numerator) / np.longdouble(odd.denominator) *
              (np.longdouble(n[a]) / np.longdouble(L[a])) ** 2 for a in range(3))
    assert abs(float(np.mean(y / x) / lam - 1)) <= 2.0 ** -55
