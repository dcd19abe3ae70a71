"""Gram product and rotation of real blocks as digit products (hub_gram, hub_rayleigh_ritz)
against 64-bit sums: sizes around the tiles of 128 and 64 columns and the steps of 16 and 512
points, odd leading dimensions, columns of very different and of extreme magnitude, constant
columns (equal digits at every point), localized columns, non-finite values.

Bound: every operand is rounded at u of its column's largest magnitude (2^-53 double, 2^-29
float: half a unit of 54 and 30 bits below the next power of two, with room), which a sum of K
terms carries as u sqrt(K) (|a|max |b| + |b|max |a|); dropped products are below v of |a|max
|b|max per term (2^-51, 2^-36); the reference is a correctly rounded sum."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F32, HUB_F64, Hub  # noqa: E402

CASES = [((5, 3, 1), 1, 0), ((7, 9, 8), 64, 0), ((8, 8, 8), 65, 3), ((16, 16, 4), 128, 1), ((13, 17, 11), 129, 0),
         ((40, 30, 9), 200, 5), ((33, 9, 17), 348, 0)]


def grid(n, prec):
    """Float blocks take the digits from 8192 points on: the third axis as often as that needs."""
    k = 1 if prec == HUB_F64 else -(-8192 // (n[0] * n[1] * n[2]))
    return n[0], n[1], n[2] * k


def check(G, A, B, prec):
    """Every entry, or (large products) the first 4 x 4 and 400 others, against a correctly
    rounded sum of the products."""
    lim = bound(A, B, prec)
    m, n = G.shape
    if m * n * A.shape[1] <= 2_000_000:
        todo = [(i, j) for i in range(m) for j in range(n)]
    else:
        rng = np.random.default_rng(1)
        todo = [(i, j) for i in range(min(4, m)) for j in range(min(4, n))] + \
            [(int(rng.integers(m)), int(rng.integers(n))) for _ in range(400)]
    for i, j in todo:
        ref = math.fsum(A[i] * B[j])
        assert abs(G[i, j] - ref) <= lim[i, j], (i, j, G[i, j], ref, lim[i, j])


def bound(A, B, prec):
    u, v = (2.0 ** -53, 2.0 ** -51) if prec == HUB_F64 else (2.0 ** -29, 2.0 ** -36)
    K = A.shape[1]
    na, nb = np.linalg.norm(A, axis=1)[:, None], np.linalg.norm(B, axis=1)[None]
    ma, mb = np.max(np.abs(A), axis=1)[:, None], np.max(np.abs(B), axis=1)[None]
    return u * K ** 0.5 * (ma * nb + mb * na) + v * K * ma * mb + 2.0 ** -50 * na * nb + 1e-320


def run(hb, A, B, ld):
    dt = hb.dtype
    def dev(M):
        P = torch.full((M.shape[0], ld), float("nan"), dtype=dt, device="cuda")
        P[:, :M.shape[1]] = torch.tensor(M, device="cuda").to(dt)
        return P
    Ad = dev(A)
    Bd = Ad if B is A else dev(B)
    G = torch.empty(A.shape[0], B.shape[0], dtype=torch.float64, device="cuda")
    hb.gram(Ad, Bd, 1.0, G)
    return G.cpu().numpy()


@pytest.mark.parametrize("prec", [HUB_F64, HUB_F32])
@pytest.mark.parametrize("n,ncol,pad", CASES)
def test_gram(n, ncol, pad, prec):
    rng = np.random.default_rng(ncol)
    n = grid(n, prec)
    Nd = n[0] * n[1] * n[2]
    np_t = np.float64 if prec == HUB_F64 else np.float32
    hb = Hub(n, (1.0, 1.1, 1.2), 6, prec=prec)
    A = rng.standard_normal((ncol, Nd)) * np.logspace(0, -12, ncol)[:, None]
    A[0] = 0.7123456789                                  # equal digits at every point
    if ncol > 2:
        A[1] *= np.exp(-np.arange(Nd) / 3.0)             # localized
        A[2] = 0.0
    A = A.astype(np_t).astype(np.float64)
    B = rng.standard_normal((max(1, ncol // 2), Nd)).astype(np_t).astype(np.float64)
    for X, Y in ((A, A), (A, B)):
        G = run(hb, X, Y, Nd + pad)
        check(G, X, Y, prec)
        if X is Y:
            assert np.array_equal(G, G.T)


@pytest.mark.parametrize("prec,tiny,huge", [(HUB_F64, 1e-290, 1e150), (HUB_F32, 1e-33, 1e33)])
def test_gram_outside_the_format(prec, tiny, huge):
    rng = np.random.default_rng(4)
    n = grid((9, 10, 11), prec)
    Nd = n[0] * n[1] * n[2]
    np_t = np.float64 if prec == HUB_F64 else np.float32
    hb = Hub(n, (1.0, 1.1, 1.2), 6, prec=prec)
    A = rng.standard_normal((5, Nd)) * np.array([1.0, tiny, huge, 1.0, 1.0])[:, None]
    A = A.astype(np_t).astype(np.float64)
    A[3, 77] = np.nan
    A[4, 5] = np.inf
    B = rng.standard_normal((3, Nd)).astype(np_t).astype(np.float64)
    G = run(hb, A, B, Nd)
    check(G[:3], A[:3], B, prec)
    assert np.all(np.isnan(G[3])) and np.all(~np.isfinite(G[4]))


@pytest.mark.parametrize("prec", [HUB_F64, HUB_F32])
@pytest.mark.parametrize("n,ncol", [((12, 10, 9), 3), ((16, 14, 12), 63), ((20, 18, 16), 130), ((48, 44, 40), 140)])
def test_rotation_through_rayleigh_ritz(n, ncol, prec):
    """With no atoms, V = 0 and columns of very different size: the rotated block is orthonormal
    and spans the block it came from."""
    rng = np.random.default_rng(ncol)
    Nd = n[0] * n[1] * n[2]
    L = tuple(0.4 * v for v in n)
    dV = 0.4 ** 3
    hb = Hub(n, L, 6, prec=prec)
    hb.set_veff(torch.tensor(rng.uniform(-1, 0, Nd), device="cuda"))
    hb.set_atoms([])
    X0 = rng.standard_normal((ncol, Nd)) * np.logspace(0, -3, ncol)[:, None]
    X = torch.tensor(X0, device="cuda").to(hb.dtype)
    X0 = X.double().cpu().numpy()
    hb.rayleigh_ritz(0, X)
    Y = X.double().cpu().numpy()
    tol = 1e-11 if prec == HUB_F64 else 2e-5             # rounding times the block's condition (about 10)
    assert np.max(np.abs(dV * Y @ Y.T - np.eye(ncol))) < tol
    # P X0 = X0 with the projector of the rotated block
    D = X0 - dV * (X0 @ Y.T) @ Y
    assert np.max(np.linalg.norm(D, axis=1) / np.linalg.norm(X0, axis=1)) < tol
