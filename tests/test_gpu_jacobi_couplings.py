"""What Rayleigh-Ritz leaves of the couplings between the orbitals of a double block: rounding, not the
threshold at which sweeps stop."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F64, Hub  # noqa: E402


@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("ncol", [2, 3, 4, 6])
def test_couplings_are_rounded_away(ncol, complex_):
    """60 random blocks per size: |<x_i|H|x_j>| <= 1e-14 of the largest diagonal.  The inner products
    here are taken in extended precision; what is left is the rounding of 720-term operands, of H x
    (about 3 times the diagonal at most) and of a rotation: some 1e-15."""
    rng = np.random.default_rng(10 * ncol + complex_)
    n, Nd = (8, 9, 10), 720
    hb = Hub(n, tuple(0.4 * m for m in n), 6, kpt=(0.1, 0.2, 0.3) if complex_ else (0.0, 0.0, 0.0), complex_=complex_,
             prec=HUB_F64)
    hb.set_veff(torch.tensor(rng.uniform(-3, 0, Nd), device="cuda"))
    hb.set_atoms([])
    dV = 0.4 ** 3
    worst = 0.0
    for _ in range(60):
        x = rng.standard_normal((ncol, Nd))
        if complex_:
            x = x + 1j * rng.standard_normal((ncol, Nd))
        X = torch.tensor(x, device="cuda")
        hb.rayleigh_ritz(0, X)
        Y = torch.empty_like(X)
        hb.apply_H(0, X, Y)
        wide = np.clongdouble if complex_ else np.longdouble
        M = np.abs((X.cpu().numpy().astype(wide).conj() @ Y.cpu().numpy().astype(wide).T) * dV).astype(float)
        d = np.diag(M).max()
        worst = max(worst, (M - np.diag(np.diag(M))).max() / d)
    assert worst <= 1e-14
