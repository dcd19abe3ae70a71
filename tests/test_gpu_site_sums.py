"""Sums of the projector inner products over bricks: float blocks against the FP64 form.

Bias: for positive values every addition inside the tensor core cuts the running sum off, by half
a unit (2^-24) on average; an accumulator takes 12 additions and its sum is below its last value
during them, so the inner products are at most 12 * 2^-24 = 7.2e-7 too small on average (32
additions in one accumulator: 1.9e-6).  A single one is off by twice that and its operands'
roundings: 2e-6."""
import numpy as np
import pytest

import workloads as w
from hubtest import make_hub

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F32, HUB_F64  # noqa: E402


@pytest.mark.parametrize("ncol", [1, 31, 33, 130])
@pytest.mark.parametrize("n", [(20, 12, 12), (28, 30, 21)])
def test_inner_products_of_positive_values(n, ncol):
    wl = w.small_test_system(n=n, natoms=12, ncol=ncol, seed=7, hub_rc=2.5, kb_rc=2.5)
    X = 0.5 + np.random.default_rng(ncol).random((ncol, wl.Nd)).astype(np.float32)
    wide = make_hub(wl, HUB_F64).project(torch.tensor(X, dtype=torch.float64, device="cuda"))
    c = make_hub(wl, HUB_F32).project(torch.tensor(X, device="cuda"))
    # rows whose function does not change sign: their inner products are the largest
    rows = np.abs(wide).mean(1) > 0.5 * np.abs(wide).mean(1).max()
    err = c[rows] / wide[rows] - 1.0
    assert abs(err.mean()) < 12 * 2.0 ** -24
    assert np.abs(err).max() < 2e-6
