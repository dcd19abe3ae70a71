"""Which form takes the Gram product of a float block (hub_gram): a few columns of a large grid stay on
CUDA cores, where they fill one tile; the digit form shows by its column maxima.  Both against 64-bit
sums: the bound is one float rounding of every product and of the partial sums (2^-24 times 16)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F32, HUB_F64, Hub  # noqa: E402


@pytest.mark.parametrize("prec,n,cols,ld_extra,digits", [
    (HUB_F32, (24, 24, 24), 1, 0, False), (HUB_F32, (24, 24, 24), 2, 0, True), (HUB_F32, (32, 32, 32), 1, 0, True),
    (HUB_F32, (60, 60, 64), 1, 0, False), (HUB_F32, (72, 72, 72), 3, 0, True), (HUB_F32, (88, 88, 84), 3, 0, False),
    (HUB_F32, (88, 88, 84), 4, 0, True), (HUB_F32, (100, 100, 100), 8, 0, False), (HUB_F32, (100, 100, 100), 64, 0, False),
    (HUB_F32, (100, 100, 100), 65, 0, True), (HUB_F32, (100, 100, 100), 8, 1, True), (HUB_F64, (100, 100, 100), 2, 0, True)])
def test_route(prec, n, cols, ld_extra, digits):
    Nd = n[0] * n[1] * n[2]
    hb = Hub(n, (1.0, 1.1, 1.2), 6, prec=prec)
    g = torch.Generator(device="cuda")
    g.manual_seed(cols)
    A = torch.randn((cols, Nd + ld_extra), generator=g, device="cuda", dtype=hb.dtype)
    G = torch.empty(cols, cols, dtype=torch.float64, device="cuda")
    hb.profile(1)
    hb.gram(A, A, 1.0, G)
    assert ("copy" in hb.profile_read()) == digits
    hb.profile(-1)
    X = A[:, :Nd].double()
    ref = X @ X.T
    norm = torch.sqrt(torch.diagonal(ref))
    u = 2.0 ** -24 if prec == HUB_F32 else 2.0 ** -50
    assert torch.max(torch.abs(G - ref) / (norm[:, None] * norm[None])).item() <= 16 * u
