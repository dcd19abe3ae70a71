"""The rotations of the subspace eigensolver leave no coupling behind: a 2 x 2 problem ends after one
sweep (hub_scf_result.jacobi_sweeps), whatever the ratio of its coupling to its gap."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F64, Hub, scf_params  # noqa: E402


@pytest.mark.parametrize("degree", [1, 2, 4, 8])
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_two_orbitals_take_one_sweep(seed, degree):
    """Two orbitals of a small box, filtered a little: coupling and gap of the projected matrix are of
    the same order after degree 1 and further apart with every degree.  One exact rotation leaves a
    coupling of a few ulp, under the threshold of 1e-13 of the diagonal."""
    rng = np.random.default_rng(seed)
    n = (8, 9, 10)
    Nd = 720
    hb = Hub(n, tuple(0.4 * m for m in n), 6, prec=HUB_F64)
    hb.set_veff(torch.tensor(rng.uniform(-3, 0, Nd), device="cuda"))
    hb.set_atoms([])
    X = torch.tensor(rng.standard_normal((2, Nd)), device="cuda")
    v0 = torch.tensor(rng.standard_normal(Nd), device="cuda")
    p = scf_params(nspin=1, ncol=2, ld=Nd, degree=degree, max_iter=5, first_passes=1, lanczos_steps=10, pulay_history=3,
                   natoms=1, pulay_beta=0.3, kT=0.05, n_elec=2.0, tol_e_atom=1e-7, tol_D=1e-4)
    hb.scf_begin(p, [X], [v0], np.zeros((1, 0, 5, 5)))
    r = hb.scf_iterate()
    assert math.isfinite(r["E"])
    assert r["jacobi_sweeps"] == 1
