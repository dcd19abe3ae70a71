"""hub_expand in the digit form, shown to have run (its own launch finds the maxima of W), for every
element type: bricks whose chunks of 16 slots all stay in shared memory and bricks with more, more
bricks than SMs, partial tiles of columns and odd rows.  Bound as for the gather and scatter of
tests/test_gpu_projector_digits.py: 16 u per term."""
import numpy as np
import pytest

import workloads as w
from hubtest import make_hub
from test_gpu_projector_digits import KPT, tables

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F32, HUB_F64  # noqa: E402

# 150 bricks with some 60 slots; 48 with some 200 (a chunk has 16; 3 or 5 of them stay)
SYSTEMS = {"few slots": dict(n=(37, 34, 24), natoms=12, seed=3, hub_rc=3.5, kb_rc=3.5),
           "many slots": dict(n=(29, 18, 14), natoms=18, seed=4, hub_rc=3.5, kb_rc=3.5),
           "three rounds": dict(n=(53, 50, 42), natoms=16, seed=5, hub_rc=4.5, kb_rc=4.5)}


@pytest.mark.parametrize("prec,cplx", [(HUB_F64, False), (HUB_F64, True), (HUB_F32, False), (HUB_F32, True)])
@pytest.mark.parametrize("name", list(SYSTEMS))
def test_expand_in_the_digit_form(name, prec, cplx):
    ncol = 130
    wl = w.small_test_system(ncol=ncol, kpt=KPT if cplx else (0, 0, 0), **SYSTEMS[name])
    _, P = tables(wl)
    u = 2.0 ** -53 if prec == HUB_F64 else 2.0 ** -24
    hb = make_hub(wl, prec, complex_=cplx)
    rng = np.random.default_rng(3)
    W = rng.standard_normal((P.shape[1], ncol)) + (1j * rng.standard_normal((P.shape[1], ncol)) if cplx else 0)
    Y = torch.zeros(ncol, wl.Nd + 3, dtype=hb.dtype, device="cuda")
    hb.profile(1)
    hb.expand(W, Y, -0.7)
    assert hb.profile_read()["scatter"][1] == 2
    hb.profile(-1)
    got = Y.cpu().numpy()
    assert np.all(got[:, wl.Nd:] == 0)
    if prec == HUB_F32:
        W = W.astype(np.complex64 if cplx else np.float32).astype(W.dtype)
    ref = -0.7 * (P @ W).T
    terms = np.count_nonzero(P, axis=1)[None, :] + 1
    bound = 16 * u * terms * np.max(np.abs(W), axis=0)[:, None] * np.max(np.abs(P))
    assert np.all(np.abs(got[:, :wl.Nd] - ref) <= bound)
