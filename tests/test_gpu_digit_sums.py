"""Sums of digit products at their largest: operands whose leading three digits are nearly full and of
one sign at every point, the others different from point to point.  A level of 512 such products
passes 2^24, where the tensor core's FP32 accumulator drops the odd units; the double forms read
theirs out every 256.  Gram product, complex gather (512 reals per brick) and scatter (480 functions
on a point).

The top 24 bits of an operand are 63, 127, 127 in base 256 (of 64 at most in the first digit), the
fourth digit is 64 to 127: x = (63 + 127/256 + 127/65536 + [0.25, 0.49)/65536) 2^k."""
import math

import numpy as np
import pytest

from oracle import hubbard as o

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F64, Hub  # noqa: E402

TOP = 63 + 127 / 256 + 127 / 65536


def full(rng, shape):
    return (TOP + rng.uniform(0.25, 0.49, shape) / 65536) / 64


class _Atom:
    """One s function, nearly flat over its sphere."""
    def __init__(self, pos, rs, rc):
        self.pos, self.kb_l, self.kb_rs, self.kb_gamma, self.kb_rc = np.asarray(pos), (0,), (rs,), (1.0,), rc
        self.hub_l, self.hub_rs, self.hub_rc, self.hub_U = -1, 1.0, 0.0, 0.0


def flat_width(grid, pos, rc, comp):
    """The width near 40000 bohr whose values have the full leading digits: over the sphere they
    differ by 2^-29 of themselves, a hundredth of the third digit's unit."""
    rs = 40000.0
    for _ in range(20):
        _, v = o.atom_function_table(grid, pos, [(0, rs)], rc)
        top = np.max(np.abs(comp(v)))
        want = (TOP + 0.45 / 65536) / 64
        m = math.frexp(top)[0]
        rs *= (m / want) ** (2 / 3)
    return rs


@pytest.mark.parametrize("nd", [(48, 48, 40), (60, 50, 33)])
def test_gram(nd):
    """Grids that leave every SM more than 512 points.  Operands are exact in 54 bits; one rounding of
    the sum and the dropped levels: 2^-50."""
    rng = np.random.default_rng(1)
    K = nd[0] * nd[1] * nd[2]
    hb = Hub(nd, (1.0, 1.1, 1.2), 6, prec=HUB_F64)
    A, B = full(rng, (3, K)), -full(rng, (2, K))
    G = torch.empty(3, 2, dtype=torch.float64, device="cuda")
    hb.gram(torch.tensor(A, device="cuda"), torch.tensor(B, device="cuda"), 1.0, G)
    G = G.cpu().numpy()
    for i in range(3):
        for j in range(2):
            ref = math.fsum(A[i] * B[j])
            assert abs(G[i, j] - ref) <= 2.0 ** -50 * abs(ref), (i, j, G[i, j] / ref - 1)


def test_complex_gather():
    """60 equal functions an eighth of a period into the next cell (phase exp(i pi / 4): real and
    imaginary parts alike), centred in the grid; 130 columns, real and imaginary parts full."""
    n, h = (32, 32, 32), 0.2
    L = tuple(h * m for m in n)
    k = (math.pi / 4 / L[0], 0.0, 0.0)
    pos = np.array([2.8 - L[0], 2.8, 2.8])
    grid = o.Grid(n, L, k)
    rs = flat_width(grid, pos, 2.5, lambda v: v.real)
    idx, P = o.atom_function_table(grid, pos, [(0, rs)], 2.5)
    hb = Hub(n, L, 6, prec=HUB_F64, complex_=True, kpt=k)
    hb.set_atoms([_Atom(pos, rs, 2.5) for _ in range(60)])
    rng = np.random.default_rng(2)
    X = full(rng, (130, 32768)) + 1j * full(rng, (130, 32768)) * np.sign(P[0, 0].imag / P[0, 0].real)
    hb.profile(1)
    C = hb.project(torch.tensor(X, device="cuda"))
    assert "copy" in hb.profile_read()              # the digit form ran
    hb.profile(-1)
    p = P[:, 0]
    for j in (0, 64, 129):
        re = math.fsum((p.real * X[j, idx].real).tolist() + (p.imag * X[j, idx].imag).tolist()) * grid.dV
        assert abs(C[0, j].real - re) <= 16 * 2.0 ** -53 * abs(re)


def test_scatter():
    """480 equal functions on one place, coefficients full."""
    n, h = (32, 32, 32), 0.2
    L = tuple(h * m for m in n)
    pos = np.array([2.8, 2.8, 2.8])
    grid = o.Grid(n, L)
    rs = flat_width(grid, pos, 2.5, lambda v: v)
    idx, P = o.atom_function_table(grid, pos, [(0, rs)], 2.5)
    hb = Hub(n, L, 6, prec=HUB_F64)
    hb.set_atoms([_Atom(pos, rs, 2.5) for _ in range(480)])
    rng = np.random.default_rng(3)
    W = full(rng, (480, 20))
    Y = torch.zeros(20, 32768, dtype=torch.float64, device="cuda")
    hb.profile(1)
    hb.expand(W, Y, 1.0)
    assert hb.profile_read()["scatter"][1] == 2     # maxima of W, then the digit form
    hb.profile(-1)
    Y = Y.cpu().numpy()
    for j in (0, 7, 19):
        s = math.fsum(W[:, j])
        assert np.max(np.abs(Y[j, idx] - P[:, 0] * s)) <= 16 * 2.0 ** -53 * s * np.max(P)
