"""The digit form of the projector gather and scatter (FP64, complex, and real float blocks on
grids whose rows are not multiples of 4), through hub_project and hub_expand, against the
oracle's tables: bricks that end inside the grid, odd rows and leading dimensions (copies of
single elements), orbital counts around the tiles of 16, 32 and 128 (two tiles in FP64), bricks that carry several
groups of functions, columns of any magnitude and non-finite values.

Bound per element: the operands are rounded at u of their column's and function's largest
magnitude (2^-53 double; float tables and blocks carry 2^-24), and so is the oracle's sum:
16 u xmax phimax dV per point of the support."""
import numpy as np
import pytest

import workloads as w
from oracle import hubbard as o
from hubtest import make_hub

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F32, HUB_F64  # noqa: E402

KPT = (0.21, -0.13, 0.34)


def tables(wl):
    g = o.Grid(wl.n, wl.L, wl.kpts[0])
    cols = []
    for a in wl.atoms:
        for ch, rc in ((list(zip(a.kb_l, a.kb_rs)), a.kb_rc), ([(a.hub_l, a.hub_rs)] if a.hub_l >= 0 else [], a.hub_rc)):
            if ch:
                idx, vals = o.atom_function_table(g, a.pos, ch, rc)
                B = np.zeros((wl.Nd, vals.shape[1]), dtype=vals.dtype)
                B[idx] = vals
                cols.append(B)
    return g, np.concatenate(cols, axis=1)


def block(wl, prec, cplx, scale=1.0, pad=0):
    rng = np.random.default_rng(9)
    X = rng.standard_normal((wl.ncol, wl.Nd)) * scale
    if cplx:
        X = X + 1j * rng.standard_normal((wl.ncol, wl.Nd)) * scale
    t = {(0, 0): np.float32, (0, 1): np.complex64, (1, 0): np.float64, (1, 1): np.complex128}[(int(prec == HUB_F64), int(cplx))]
    Xp = np.full((wl.ncol, wl.Nd + pad), np.nan, dtype=t)
    Xp[:, :wl.Nd] = X.astype(t)
    return Xp


# crowded cells: the digit form is the one chosen (launch rule by function values and columns)
SYSTEMS = {
    "even-rows": dict(n=(20, 12, 12), natoms=14, seed=7, hub_rc=2.5, kb_rc=2.5),
    "odd-rows": dict(n=(13, 10, 9), natoms=18, seed=21, hub_rc=2.5, kb_rc=2.5),
    "two-mod-4": dict(n=(18, 11, 6), natoms=20, seed=5, hub_rc=2.5, kb_rc=2.5),
    "crowded": dict(n=(15, 16, 17), natoms=12, seed=21, hub_rc=2.5, kb_rc=2.5),
    "thin": dict(n=(3, 5, 40), natoms=2, seed=8, hub_rc=0.8, kb_rc=0.8),
}


@pytest.mark.parametrize("name,ncol,pad,prec,cplx", [
    ("even-rows", 45, 0, HUB_F64, False), ("odd-rows", 130, 3, HUB_F64, False), ("two-mod-4", 129, 1, HUB_F64, False),
    ("crowded", 17, 0, HUB_F64, False), ("crowded", 1, 2, HUB_F64, False), ("thin", 1, 5, HUB_F64, False),
    ("even-rows", 45, 0, HUB_F64, True), ("odd-rows", 130, 3, HUB_F64, True), ("two-mod-4", 129, 1, HUB_F64, True),
    ("crowded", 17, 0, HUB_F64, True), ("thin", 1, 5, HUB_F64, True),
    ("even-rows", 45, 0, HUB_F32, True), ("odd-rows", 120, 3, HUB_F32, True), ("two-mod-4", 128, 1, HUB_F32, True),
    ("crowded", 17, 0, HUB_F32, True), ("thin", 1, 5, HUB_F32, True),
    ("odd-rows", 120, 3, HUB_F32, False), ("two-mod-4", 128, 1, HUB_F32, False), ("crowded", 17, 0, HUB_F32, False)])
def test_gather_and_scatter(name, ncol, pad, prec, cplx):
    wl = w.small_test_system(ncol=ncol, kpt=KPT if cplx else (0, 0, 0), **SYSTEMS[name])
    g, P = tables(wl)
    u = 2.0 ** -53 if prec == HUB_F64 else 2.0 ** -24
    hb = make_hub(wl, prec, complex_=cplx)
    X = block(wl, prec, cplx, pad=pad)
    Xd = torch.tensor(X, device="cuda")
    Xe = X[:, :wl.Nd].astype(np.complex128 if cplx else np.float64)
    ref = g.dV * (P.conj().T @ Xe.T)
    hb.profile(1)
    got = hb.project(Xd)
    # the column maxima show that the digit form ran ("thin" and single columns: either form)
    assert "copy" in hb.profile_read() or name == "thin" or ncol == 1
    hb.profile(-1)
    pts = np.count_nonzero(P, axis=0)[:, None]
    phimax = np.max(np.abs(P), axis=0)[:, None]
    assert np.all(np.abs(got - ref) <= 16 * u * g.dV * np.max(np.abs(Xe), axis=1) * phimax * pts)
    # scatter of random coefficients; the padding stays as it was
    rng = np.random.default_rng(3)
    W = rng.standard_normal((P.shape[1], ncol)) + (1j * rng.standard_normal((P.shape[1], ncol)) if cplx else 0)
    W = W.astype(X.dtype).astype(Xe.dtype)
    hb.expand(W, Xd, -0.7)
    refY = Xe - 0.7 * (P @ W).T
    out = Xd.cpu().numpy()
    assert np.all(np.isnan(out[:, wl.Nd:]))
    terms = np.count_nonzero(P, axis=1)[None, :] + 1
    bound = 16 * u * (np.abs(Xe) + terms * np.max(np.abs(W), axis=0)[:, None] * np.max(np.abs(P)))
    assert np.all(np.abs(out[:, :wl.Nd] - refY) <= bound)


@pytest.mark.parametrize("prec,cplx,tiny,huge", [(HUB_F64, False, 1e-280, 1e280), (HUB_F64, True, 1e-280, 1e280),
                                                 (HUB_F32, True, 1e-30, 1e30)])
def test_columns_outside_the_format(prec, cplx, tiny, huge):
    """Columns far from 1, a zero column, and one NaN and one infinity: each reaches only the
    functions (gather) and the points (scatter) it belongs to."""
    wl = w.small_test_system(ncol=96, kpt=KPT if cplx else (0, 0, 0), **SYSTEMS["odd-rows"])
    g, P = tables(wl)
    u = 2.0 ** -53 if prec == HUB_F64 else 2.0 ** -24
    hb = make_hub(wl, prec, complex_=cplx)
    X = block(wl, prec, cplx, scale=np.tile([1.0, tiny, huge, 0.0, 1.0, 1.0], 16)[:, None])
    # a point inside some functions and outside others
    inside = np.count_nonzero(P, axis=1)
    pt = int(np.argmin(np.where(inside > 0, inside, 10 ** 9)))
    X[4, pt] = np.nan
    X[5, pt] = np.inf
    Xe = X.astype(np.complex128 if cplx else np.float64)
    hb.profile(1)
    got = hb.project(torch.tensor(X, device="cuda"))
    assert "copy" in hb.profile_read()
    hb.profile(-1)
    hit = np.abs(P[pt]) > 0
    for j in (4, 5):
        assert np.all(~np.isfinite(got[hit, j])) and np.all(np.isfinite(got[~hit, j]))
    rest = Xe.copy()
    rest[4:6, pt] = 0
    with np.errstate(under="ignore"):
        ref = g.dV * (P.conj().T @ rest.T)
    pts = np.count_nonzero(P, axis=0)[:, None]
    bound = 16 * u * g.dV * np.max(np.abs(rest), axis=1) * np.max(np.abs(P), axis=0)[:, None] * pts
    ok = np.ones(ref.shape, dtype=bool)
    ok[np.ix_(hit, [4, 5])] = False
    assert np.all((np.abs(got - ref) <= bound)[ok])
    # scatter: W with a NaN in one row, and rows of the extreme magnitudes
    rng = np.random.default_rng(3)
    W = rng.standard_normal((P.shape[1], 96)) * np.tile([1.0, tiny, huge, 0.0, 1.0, 1.0], 16) + (0j if cplx else 0)
    row = int(np.argmin(pts[:, 0]))
    W[row, 4] = np.nan
    Y0 = block(wl, prec, cplx)
    Yd = torch.tensor(Y0, device="cuda")
    hb.expand(W, Yd, 1.0)
    out = Yd.cpu().numpy()
    hitp = np.abs(P[:, row]) > 0
    assert np.all(~np.isfinite(out[4, hitp])) and np.all(np.isfinite(out[4, ~hitp]))
    Wf = np.where(np.isfinite(W), W, 0).astype(Y0.dtype).astype(Xe.dtype)
    refY = Y0.astype(Xe.dtype) + (P @ Wf).T
    terms = np.count_nonzero(P, axis=1)[None, :] + 1
    bound = 16 * u * (np.abs(Y0) + terms * np.max(np.abs(Wf), axis=0)[:, None] * np.max(np.abs(P)))
    bad = np.zeros(out.shape, dtype=bool)
    bad[4, hitp] = True
    assert np.all((np.abs(out - refY) <= bound) | bad)
