"""H psi of the precision form with projectors and states of very different scale, whose products are
ordinary numbers: the result depends on the scales only through FP32's range.  Against the oracle, 1e-6 per
band (the precision form's bar); FP32 holds the scaled operands, the projections and the result."""
import numpy as np
import pytest

import qm_synth as S
from oracle import hamiltonian as OH

from cases import band_rel_err, make_case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2308_07277_gb300 as Q
    return Q


@pytest.mark.parametrize("nb", [4, 96])          # FP32 on the CUDA cores, tensor cores
@pytest.mark.parametrize("fb,fp", [(1e36, 1e-35), (1e-34, 1e33), (1e16, 1e16), (1e-15, 1e-15)])
def test_scales(Q, nb, fb, fp):
    cell = S.cubic_si8(15.0, nbnd=nb, kpts=[[0.25, 0.25, 0.25]])
    c = make_case(cell, 0)
    beta, psi = (c["beta"] * fb).astype(np.complex64), (c["psi"] * fp).astype(np.complex64)
    D = c["D"] / fb
    g = Q.qm_gspace_create(cell.lattice, cell.kpts, cell.ecut_ha, cell.grid)
    try:
        out = Q.qm_hpsi(g, 0, torch.from_numpy(psi).cuda(), torch.from_numpy(c["v"]).cuda(), torch.from_numpy(beta).cuda(),
                        torch.from_numpy(np.ascontiguousarray(D)).cuda(), prec="mixed").cpu().numpy()
    finally:
        Q.qm_gspace_destroy(g)
    want = OH.hpsi_fft(psi.astype(complex), c["gs"], c["v"], beta.astype(complex), D)
    assert np.isfinite(out).all()
    assert band_rel_err(out, want).max() <= 1e-6
