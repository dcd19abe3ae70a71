"""A handle without room for what only makes products faster (hub_set_memory_limit: its allocations
fail as cudaMalloc does on a full device): every call that fits in some form gives its result, in
that form, and nothing is tried again on every call."""
import numpy as np
import pytest

import workloads as w
from hubtest import make_hub, rel

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F32, HUB_F64, Hub, HubError, batch_filter  # noqa: E402

KPT = (0.21, -0.13, 0.34)
TOL = {HUB_F64: 1e-12, HUB_F32: 1e-4}       # two forms of the same sums of a few hundred terms


def crowded(cplx, prec, ncol=96):
    wl = w.small_test_system(n=(13, 10, 9), natoms=18, seed=21, hub_rc=2.5, kb_rc=2.5, ncol=ncol, kpt=KPT if cplx else (0, 0, 0))
    hb = make_hub(wl, prec, complex_=cplx)
    hb.set_occupation_matrix(0, wl.D0[0])
    X = torch.tensor(wl.orbitals(complex_=cplx), device="cuda").to(hb.dtype)
    return wl, hb, X


def forms(hb, call):
    hb.profile(1)
    out = call()
    kinds = hb.profile_read()
    hb.profile(-1)
    return out, "copy" in kinds, kinds


def message(hb):
    return hb.lib.hub_last_error(hb.h)


@pytest.mark.parametrize("cplx,prec", [(False, HUB_F64), (True, HUB_F64), (True, HUB_F32)])
def test_no_room_for_the_digit_tables(cplx, prec):
    wl, hb, X = crowded(cplx, prec)
    tables = hb.memory_held()
    assert tables > 1 << 20
    ref, digits, _ = forms(hb, lambda: hb.project(X))
    assert digits
    hb.close()
    _, hb, X = crowded(cplx, prec)
    hb.set_memory_limit(1)
    hb.set_atoms(wl.atoms)
    assert hb.memory_held() == 8 * wl.Nd     # the copy of V
    with pytest.raises(HubError) as e:
        hb.project(X)
    assert e.value.code == -2                # HUB_ENOMEM
    hb.set_memory_limit(tables - 1)
    hb.set_atoms(wl.atoms)
    got, digits, _ = forms(hb, lambda: hb.project(X))
    assert not digits and rel(got, ref) < TOL[prec]
    hb.set_memory_limit(0)
    hb.set_atoms(wl.atoms)
    got, digits, _ = forms(hb, lambda: hb.project(X))
    assert digits and rel(got, ref) < TOL[prec]


@pytest.mark.parametrize("cplx,prec", [(False, HUB_F64), (True, HUB_F64), (True, HUB_F32)])
def test_workspaces_take_the_room_of_the_digits(cplx, prec):
    """Room for the tables and little more, from none to plenty: H X is right in all of them, first by
    giving the tables back, then without the gather's digit workspace, then in the digit form."""
    wl, hb, X = crowded(cplx, prec)
    Y = torch.empty_like(X)
    hb.apply_H(0, X, Y)
    ref = Y.cpu().numpy()
    hb.close()
    seen = set()
    for extra in [0] + [1 << k for k in range(10, 27)]:
        _, hb, X = crowded(cplx, prec)
        tables = hb.memory_held()
        hb.set_memory_limit(tables + extra)
        for _ in range(2):                   # the second call finds everything as the first left it
            Y.zero_()
            hb.apply_H(0, X, Y)
            assert rel(Y.cpu().numpy(), ref) < TOL[prec], extra
            assert hb.memory_held() <= tables + extra and message(hb) == b""
        _, digits, _ = forms(hb, lambda: hb.project(X))
        seen.add((hb.memory_held() < tables, digits))
        hb.close()
    assert seen == {(True, False), (False, False), (False, True)} or seen == {(True, False), (False, True)}


@pytest.mark.parametrize("prec", [HUB_F64, HUB_F32])
def test_products_with_less_room(prec):
    """Gram product and Rayleigh-Ritz of 200 orbitals on 43,200 points: all digits at once, in several
    panels, and (FP64, whose partial sums take less room) on CUDA cores."""
    n = (40, 30, 36)
    Nd = n[0] * n[1] * n[2]
    rng = np.random.default_rng(1)
    X0 = torch.tensor(rng.standard_normal((200, Nd)), device="cuda")
    L = tuple(0.4 * m for m in n)
    out, panels, cores = {}, set(), False
    for limit in [0, 400 << 20, 120 << 20, 60 << 20] + ([28 << 20] if prec == HUB_F64 else []):
        hb = Hub(n, L, 6, prec=prec)
        hb.set_veff(torch.full((Nd,), -0.5, dtype=torch.float64, device="cuda"))
        hb.set_atoms([])
        hb.set_memory_limit(limit + hb.memory_held() if limit else 0)
        X = X0.clone().to(hb.dtype)
        G = torch.empty(200, 200, dtype=torch.float64, device="cuda")
        held = []
        for _ in range(2):
            _, digits, kinds = forms(hb, lambda: hb.gram(X, X, 1.0, G))
            held.append(hb.memory_held())
            assert message(hb) == b""
        assert held[0] == held[1]
        panels.add(kinds["gram"][1] if digits else 0)
        cores |= not digits
        # on CUDA cores the partial sums alone take 26 MB: no room for the rest of Rayleigh-Ritz
        eig = hb.rayleigh_ritz(0, X, torch.empty_like(X)) if limit != 28 << 20 else out[0][1]
        out[limit] = (G.cpu().numpy(), np.asarray(eig))
        hb.close()
    for G, eig in out.values():
        assert rel(G, out[0][0]) < TOL[prec] and rel(eig, out[0][1]) < TOL[prec]
    assert 1 in panels and max(panels) > 1 and cores == (prec == HUB_F64)


def test_batched_filter_without_room():
    """Two systems in one graph, one of which gives its digit tables back while it is sized."""
    res = {}
    for extra in (None, 1 << 16, 1 << 21):
        sysm = [crowded(True, HUB_F64, 40), crowded(True, HUB_F64, 40)]
        if extra is not None:
            sysm[0][1].set_memory_limit(sysm[0][1].memory_held() + extra)
        hubs, Xs = [s[1] for s in sysm], [s[2] for s in sysm]
        keep = [x.clone() for x in Xs]
        for _ in range(2):
            for x, k in zip(Xs, keep):
                x.copy_(k)
            batch_filter(hubs, [0, 0], Xs, 5, [10.0] * 2, [150.0] * 2, [-5.0] * 2)
        res[extra] = [x.cpu().numpy() for x in Xs]
        for h in hubs:
            h.close()
    for extra in (1 << 16, 1 << 21):
        for a, b in zip(res[extra], res[None]):
            assert rel(a, b) < 1e-12
