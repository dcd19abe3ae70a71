"""The gradient of float blocks behind the forces: the staged rows along x and the marched lines
along y and z against the general kernel's order of sums, through hub_hubbard_forces and the CPU
oracle.  Sizes: lines cut into chunks (few columns, long axes), ragged tails of the 4-point batches
and of the 256 lines of a CTA, axes shorter than the stencil's 6 points, rows longer than the staged
24 KB (general kernel), another order (general kernel), real and Bloch.

Tolerance: float gradient and inner products of float orbitals, 1e-4 of the norm (24-bit
significands, sums of a few thousand terms)."""
import numpy as np
import pytest

import workloads as w
from oracle import hubbard as o
from hubtest import make_hub, oracle_ham, to_dev, rel

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F32  # noqa: E402


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n,ncol,order", [((9, 61, 50), 2, 6), ((50, 9, 98), 1, 6), ((3, 20, 5), 4, 6), ((33, 16, 25), 9, 6),
                                          ((17, 4, 73), 3, 6), ((33, 16, 25), 3, 4), ((6200, 3, 2), 1, 6)])
def test_forces_of_float_blocks(n, ncol, order, cplx):
    wl = w.small_test_system(n=n, ncol=ncol, natoms=2, hub_rc=2.0, kb_rc=1.5, kpt=(0.21, -0.13, 0.34) if cplx else (0, 0, 0))
    wl.fd_half_order = order
    ct = np.complex64 if cplx else np.float32
    X = wl.orbitals(complex_=cplx).astype(ct).astype(np.complex128 if cplx else np.float64)
    f = np.linspace(1.0, 0.1, ncol)
    D = wl.D0[0].astype(np.complex128 if cplx else np.float64)
    ref_hub = o.hubbard_forces(oracle_ham(wl, D=D), X.T, f, 0.7)
    ref = np.zeros((len(wl.atoms), 3))
    ref[[i for i, a in enumerate(wl.atoms) if a.hub_l >= 0]] = ref_hub
    hb = make_hub(wl, HUB_F32)
    hb.set_occupation_matrix(0, D)
    F = hb.hubbard_forces(0, to_dev(X, hb.dtype), f, 0.7)
    assert np.max(np.abs(ref)) > 0
    assert rel(F, ref) < 1e-4
