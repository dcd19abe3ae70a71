"""Which blocks Rayleigh-Ritz takes (HUB_ENOTSPD): every positive pivot of the Gram matrix, and none
of a block that has a column twice, wherever the two stand in the blocks of 32 of the factorization."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F32, HUB_F64, Hub, HubError  # noqa: E402

N, H = (16, 16, 8), 0.5                    # dV = 1/8, 2048 points: the norm of +-1 is 2^8


def make(prec, cplx):
    hb = Hub(N, tuple(H * m for m in N), 6, prec=prec, complex_=cplx, kpt=(0.1, 0.2, 0.3) if cplx else None)
    hb.set_veff(torch.zeros(2048, dtype=torch.float64, device="cuda"))
    hb.set_atoms([])
    return hb


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("at", [1, 31, 32, 40, 64])
def test_a_small_positive_pivot_is_accepted(at, cplx):
    """Rows of a Hadamard matrix, column `at` = column 0 + 2^-25 of another row: every sum is exact in
    any order, the square root of 2^8 and the multiplier 1 too, and the pivot is 2^-50 of its diagonal
    element (which is 1 + 2^-50)."""
    h = np.array([[1.0]])
    while h.shape[0] < 2048:
        h = np.block([[h, h], [h, -h]])
    X = h[:66].copy()
    X[at] = X[0] + 2.0 ** -25 * h[100]
    hb = make(HUB_F64, cplx)
    eig = hb.rayleigh_ritz(0, torch.tensor(X, device="cuda").to(hb.dtype))
    assert np.all(np.isfinite(eig))


@pytest.mark.parametrize("prec", [HUB_F64, HUB_F32])
@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("i,j", [(0, 1), (3, 31), (0, 32), (5, 40), (33, 69), (31, 68), (40, 41)])
def test_a_column_twice_is_refused(i, j, cplx, prec):
    """Random columns: the second pivot must not depend on the rounding of the first."""
    hb = make(prec, cplx)
    rng = np.random.default_rng(100 * i + j)
    for _ in range(4):
        X = rng.standard_normal((70, 2048)) + (1j * rng.standard_normal((70, 2048)) if cplx else 0)
        X[j] = X[i]
        with pytest.raises(HubError) as e:
            hb.rayleigh_ritz(0, torch.tensor(X, device="cuda").to(hb.dtype))
        assert e.value.code == -4
