"""Complex float stencil on grids whose halo wraps around the cell once or more: against the FP64
form of the same call.  Bound: 13 sums per axis of terms that add up to at most the kinetic bound
(8 / h^2 in all) times the largest element, each rounded to 2^-24, and V, below it: 2^-20 of
(24 / h^2) max |x|."""
import numpy as np
import pytest

import workloads as w
from hubtest import make_hub

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F32, HUB_F64  # noqa: E402


@pytest.mark.parametrize("n", [(2, 3, 2), (4, 5, 3), (6, 17, 13), (18, 15, 7), (34, 33, 29)])
@pytest.mark.parametrize("ncol", [1, 3])
def test_wrapped_halos(n, ncol):
    wl = w.small_test_system(n=n, ncol=ncol, kpt=(0.31, -0.17, 0.23), natoms=1, hub_rc=0.5, kb_rc=0.5)
    g = np.random.default_rng(4)
    X = (g.standard_normal((ncol, wl.Nd)) + 1j * g.standard_normal((ncol, wl.Nd))).astype(np.complex64)
    out = []
    for prec, t in ((HUB_F64, torch.complex128), (HUB_F32, torch.complex64)):
        x = torch.tensor(X, device="cuda").to(t)
        y = torch.empty_like(x)
        make_hub(wl, prec).apply_H(0, x, y)
        out.append(y.cpu().numpy().astype(np.complex128))
    h = min(wl.L[a] / n[a] for a in range(3))
    assert np.abs(out[1] - out[0]).max() < 2.0 ** -20 * 24 / h ** 2 * np.abs(X).max()
