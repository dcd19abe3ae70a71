"""Digit gather with whole bricks as groups (cells of many bricks): up to 128 float or 64 double slots
in one accumulator, several instructions per digit.  Many columns at once (digits) against one column
at a time (the point-major form).

Bound: operands are rounded to half a unit of the largest of their column and function; for the s
functions a sum's terms are a twelfth of the largest on average, so 24 units for both operands, and
the other form's sums round as often: 64 units (2^-53; 2^-24 in float) of the largest inner product."""
import numpy as np
import pytest

import workloads as w
from hubtest import make_hub

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F32, HUB_F64  # noqa: E402


@pytest.mark.parametrize("prec,cplx", [(HUB_F64, False), (HUB_F64, True), (HUB_F32, True)])
@pytest.mark.parametrize("natoms", [30, 90])
def test_groups_of_whole_bricks(prec, cplx, natoms):
    wl = w.small_test_system(n=(72, 72, 66), ncol=130, natoms=natoms, seed=11, kpt=(0.2, -0.1, 0.3) if cplx else (0, 0, 0),
                             hub_rc=5.0, kb_rc=2.5)
    g = np.random.default_rng(natoms)
    X = 0.5 + g.random((wl.ncol, wl.Nd))
    if cplx:
        X = X + 1j * g.random((wl.ncol, wl.Nd))
    X = torch.tensor(X, device="cuda")
    if prec == HUB_F32:
        X = X.to(torch.complex64)
    hub = make_hub(wl, prec)
    many = hub.project(X)
    for j in (0, 63, 127, 129):
        one = hub.project(X[j:j + 1].contiguous())[:, 0]
        assert np.abs(many[:, j] - one).max() < 64 * (2.0 ** -53 if prec == HUB_F64 else 2.0 ** -24) * np.abs(one).max()
