"""A denormal coefficient in hub_expand, of a function so large that its product with it is not: the
digit form's scales come from normal numbers, and a denormal one must not be read as if it had a hidden
bit.  A function of width rs about a grid point has the value N Y00 ~ rs^-3/2 there and zero at all
other points."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F32, HUB_F64, Hub  # noqa: E402


class _Atom:
    def __init__(self, pos, rs, rc):
        self.pos, self.kb_l, self.kb_rs, self.kb_gamma, self.kb_rc = np.asarray(pos), (0,), (rs,), (1.0,), rc
        self.hub_l, self.hub_rs, self.hub_rc, self.hub_U = -1, 1.0, 0.0, 0.0


# peak: log2 of the large function's value; top, tiny: log2 of the other coefficients and of the denormal one
@pytest.mark.parametrize("prec,cplx,peak,top,tiny", [(HUB_F64, False, 100, -885, -1074), (HUB_F64, True, 100, -885, -1070),
                                                     (HUB_F32, True, 40, -78, -149)])
def test_denormal_coefficients(prec, cplx, peak, top, tiny):
    n, h = (32, 32, 32), 0.25                # exact: the large function's atom is on its grid point to the last bit
    L = tuple(h * m for m in n)
    rs = (2.0 ** peak / 0.4) ** (-2.0 / 3.0)
    hb = Hub(n, L, 6, prec=prec, complex_=cplx, kpt=(0.1, 0.2, 0.3) if cplx else None)
    at = (14, 15, 13)
    hb.set_atoms([_Atom((3.4, 3.4, 3.4), 0.8, 2.5) for _ in range(200)] + [_Atom([h * m for m in at], rs, 0.6)])
    W = np.full((201, 128), 2.0 ** top, dtype=complex if cplx else float)
    Y = torch.zeros(128, 32768, dtype=hb.dtype, device="cuda")
    W[200] = 1.0
    hb.expand(W, Y, 1.0)
    assert 2.0 ** (peak - 1) < torch.max(torch.abs(Y)).item() < 2.0 ** (peak + 1)
    Y.zero_()
    W[200] = 0.0
    hb.expand(W, Y, 1.0)
    Y0 = Y.cpu().numpy()
    W[200] = 2.0 ** tiny
    Y.zero_()
    hb.profile(1)
    hb.expand(W, Y, 1.0)
    assert hb.profile_read()["scatter"][1] == 2      # maxima of W, then the digit form
    hb.profile(-1)
    Y1 = Y.cpu().numpy()
    # 200 functions of at most 1; the added product is 2^(peak + tiny), rounded or left out
    u = 2.0 ** -53 if prec == HUB_F64 else 2.0 ** -24
    bound = 16 * u * 200 * 2.0 ** top
    assert 2.0 ** (peak + tiny) < bound < 2.0 ** (peak + (-1022 if prec == HUB_F64 else -126))
    assert np.max(np.abs(Y1 - Y0)) <= bound
