"""The conjugate-gradient solves behind hub_hartree and hub_kerker (fixed-point stencil, graph of 16
iterations after the first 16) against the exact inverse of the FD operator in Fourier space: odd
grids, axes shorter than the stencil, every order, handles of every type, warm starts, a wide range
of magnitudes, iteration limits on both sides of the graph.

Bound: a residual of tol |b| is an error of at most tol |b| / (smallest eigenvalue); rounding adds
some 1e-14 of cond(A) |V|, below tol for these grids."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F32, HUB_F64, Hub, HubError  # noqa: E402

H = 0.3


def symbol(n, order):
    """-Lap_h in Fourier space (n = (n1, n2, n3), x fastest)."""
    lam = 0.0
    for ax, m in enumerate(n):
        k = 2 * np.pi * np.arange(m) / m
        s = np.zeros(m)
        for p in range(1, order + 1):
            c = 2 * (-1) ** (p + 1) * math.factorial(order) ** 2 / (p * p * math.factorial(order - p) * math.factorial(order + p))
            s += c * (2 - 2 * np.cos(k * p))
        shape = [1, 1, 1]
        shape[2 - ax] = m
        lam = lam + (s / H ** 2).reshape(shape)
    return lam


def solve(n, order, rhs, lam_inv):
    f = np.fft.fftn(rhs.reshape(n[2], n[1], n[0])) * lam_inv
    return np.fft.ifftn(f).real.reshape(-1)


@pytest.mark.parametrize("prec,cplx", [(HUB_F64, False), (HUB_F32, False), (HUB_F64, True), (HUB_F32, True)])
@pytest.mark.parametrize("n,order,scale", [((12, 12, 12), 6, 1.0), ((5, 4, 7), 6, 1e-100), ((33, 9, 17), 6, 1e100), ((40, 37, 3), 2, 1.0),
                                           ((65, 24, 18), 4, 1e-9)])
def test_hartree_and_kerker(n, order, scale, prec, cplx):
    rng = np.random.default_rng(order + n[0])
    Nd = n[0] * n[1] * n[2]
    hb = Hub(n, tuple(H * m for m in n), order, prec=prec, complex_=cplx)
    rho = scale * rng.standard_normal(Nd)
    lam = symbol(n, order)
    small = np.min(lam[lam > 1e-9 * lam.max()])
    inv = np.where(lam > 1e-9 * lam.max(), 1 / np.where(lam == 0, 1, lam), 0.0)
    b = 4 * np.pi * (rho - rho.mean())
    ref = solve(n, order, b / scale, inv) * scale
    tol = 1e-11
    V = torch.zeros(Nd, dtype=torch.float64, device="cuda")
    it, eh = hb.hartree(torch.tensor(rho, device="cuda"), V, tol=tol)
    nrm = np.linalg.norm(b / scale)
    assert it % 16 == 0
    assert np.linalg.norm((V.cpu().numpy() - ref) / scale) <= 2 * tol * nrm / small
    it2, _ = hb.hartree(torch.tensor(rho, device="cuda"), V, tol=10 * tol)          # a warm start is done
    assert it2 <= 16
    k2 = 0.64
    z = torch.zeros(Nd, dtype=torch.float64, device="cuda")
    hb.kerker(torch.tensor(rho, device="cuda"), z, 0.8, tol=tol)
    zref = solve(n, order, rho / scale, lam / (lam + k2)) * scale
    lr = np.linalg.norm(solve(n, order, rho / scale, lam))
    assert np.linalg.norm((z.cpu().numpy() - zref) / scale) <= 2 * tol * lr / k2


@pytest.mark.parametrize("limit", [1, 15, 16, 17, 40])
def test_iteration_limit(limit):
    n = (30, 28, 26)
    hb = Hub(n, tuple(H * m for m in n), 6, prec=HUB_F64)
    rho = torch.tensor(np.random.default_rng(1).standard_normal(n[0] * n[1] * n[2]), device="cuda")
    V = torch.zeros_like(rho)
    with pytest.raises(HubError):
        hb.hartree(rho, V, tol=1e-12, max_iter=limit)
    # non-finite densities end at once and leave nothing behind (b . b compares false)
    hb.hartree(rho * float("nan"), V * 0, tol=1e-12)
    it, _ = hb.hartree(rho, torch.zeros_like(rho), tol=1e-10)   # the handle is as good as before
    assert it > 32
