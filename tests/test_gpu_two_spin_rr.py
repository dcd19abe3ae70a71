"""Both spins of a k-point in one Rayleigh-Ritz (hub_kscf_run with two spins) against one spin alone,
for odd and even orbital counts: the second spin's matrices follow the first's in one buffer, and
complex ones are read 16 bytes at a time."""
import numpy as np
import pytest

import workloads as w
from hubtest import to_dev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_23612_gb300 import HUB_F64  # noqa: E402
from paper_2507_23612_gb300.kpoint_scf import KpointSCF  # noqa: E402


@pytest.mark.parametrize("kpt", [(0.0, 0.0, 0.0), (0.3, -0.2, 0.25)], ids=["gamma", "bloch"])
@pytest.mark.parametrize("ncol", [3, 5, 8, 33])
def test_two_spins_agree_with_one(ncol, kpt):
    wl = w.small_test_system(n=(12, 10, 14), ncol=ncol, natoms=2, seed=11)
    eig = {}
    for ns in (1, 2):
        scf = KpointSCF(wl, [kpt], [1.0], HUB_F64)
        try:
            X = [[to_dev(wl.orbitals(complex_=any(kpt)), scf.hubs[0].dtype)] for _ in range(ns)]
            v = [[to_dev(wl.lanczos_start(complex_=any(kpt)), scf.hubs[0].dtype)] for _ in range(ns)]
            eig[ns] = scf.run(X, v, np.stack([wl.D0[0]] * ns), n_elec=0.9 * ns, kT=0.01, degree=6, max_iter=1)["eig"]
        finally:
            scf.close()
    # the same operations on the same numbers, up to the grouping of pairs in the eigensolver
    tol = 64 * ncol * 2.0 ** -52 * max(1.0, np.max(np.abs(eig[1][0][0])))
    for s in range(2):
        assert np.max(np.abs(eig[2][s][0] - eig[1][0][0])) <= tol
