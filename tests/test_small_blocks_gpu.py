"""Davidson solves whose correction blocks have sizes around the limits of the small
orthonormalisation kernels (16 and 32 vectors per block, 64-row subspace matrices), against the dense
eigensolver: eigenvalues to 1e-10 of the spectrum's lower end (residual 1e-8 squared over a gap is
below it), the vectors orthonormal to 1e-11."""
import numpy as np
import pytest

import qm_synth as S
from oracle import hamiltonian as OH

from cases import make_case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2308_07277_gb300 as Q
    return Q


@pytest.mark.parametrize("nb", [1, 15, 16, 17, 32, 33])
def test_block_sizes(Q, nb):
    cell = S.cubic_si8(10.0, nbnd=nb, kpts=[[0.25, 0.25, 0.25]])
    c = make_case(cell, 0)
    ev = np.linalg.eigvalsh(OH.dense_h(c["gs"], c["v"], c["beta"], c["D"]))[:nb]
    g = Q.qm_gspace_create(cell.lattice, cell.kpts, cell.ecut_ha, cell.grid)
    try:
        psi, v, beta, D = (torch.from_numpy(np.ascontiguousarray(c[k])).cuda() for k in ("psi", "v", "beta", "D"))
        eig, info = Q.qm_davidson(g, 0, psi, v, beta, D, tol=1e-8, max_iter=300)
        X = psi.cpu().numpy()
    finally:
        Q.qm_gspace_destroy(g)
    assert info["converged"], info
    assert np.abs(eig - ev).max() <= 1e-10
    assert np.abs(X @ X.conj().T - np.eye(nb)).max() <= 1e-11
