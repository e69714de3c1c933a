"""The precision form's nonlocal part with few projectors: on the CUDA cores up to 16, with the small terms of
the split products in accumulators of their own up to 48, together with the main ones above; one to several
row tiles of bands, projectors split on the call or prepared, against the oracle with the precision form's bars
(1e-6 per band, 5e-6 element-wise of the band's largest element).

And its error beside that of FP32 arithmetic throughout (qm_hpsi_noalloc: the same FFT path, FP32 multiply-adds in
the projector products): at most sqrt(2) times that, i.e. the split products on their own are no worse than all of
the FP32 form."""
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


def _run(Q, cell, c, beta, D, prepared, noalloc=False):
    psi = torch.from_numpy(c["psi"].astype(np.complex64)).cuda()
    g = Q.qm_gspace_create(cell.lattice, cell.kpts, cell.ecut_ha, cell.grid)
    try:
        tb, td, v = torch.from_numpy(beta).cuda(), torch.from_numpy(np.ascontiguousarray(D)).cuda(), torch.from_numpy(c["v"]).cuda()
        if prepared:
            Q.qm_hpsi_prepare(g, 0, tb)
        out = (Q.qm_hpsi_noalloc if noalloc else Q.qm_hpsi)(g, 0, psi, v, tb, td, out=torch.empty_like(psi), prec="mixed")
        return out.cpu().numpy()
    finally:
        Q.qm_gspace_destroy(g)


def _want(c, beta, D):
    return OH.hpsi_fft(c["psi"].astype(np.complex64).astype(complex), c["gs"], c["v"], beta.astype(complex), D)


@pytest.mark.parametrize("prepared", [False, True])
@pytest.mark.parametrize("ecut", [12.0, 20.0])           # rows that find their scale in the splitting kernel, longer ones
@pytest.mark.parametrize("nproj,nb", [(1, 7), (16, 3), (16, 130), (17, 64), (17, 65), (33, 63), (48, 40), (48, 129), (48, 300),
                                      (49, 40), (64, 129)])
def test_few_projectors(Q, nproj, nb, ecut, prepared):
    cell = S.cubic_si8(ecut, nbnd=nb, reps=(2, 1, 1), kpts=[[0.25, -0.25, 0.25]])
    c = make_case(cell, 0)
    beta, D = c["beta"][:nproj].astype(np.complex64), c["D"][:nproj]
    out, want = _run(Q, cell, c, beta, D, prepared), _want(c, beta, D)
    assert band_rel_err(out, want).max() <= 1e-6
    assert (np.abs(out - want).max(axis=1) <= 5e-6 * np.abs(want).max(axis=1)).all()


@pytest.mark.parametrize("nb", [56, 90])
def test_error_beside_fp32_arithmetic(Q, nb):
    cell = S.cubic_si8(15.0, nbnd=nb, kpts=[[0.25, -0.25, 0.25]])
    c = make_case(cell, 0)
    beta, D = c["beta"].astype(np.complex64), c["D"]
    want = _want(c, beta, D)
    rms = [np.sqrt((band_rel_err(_run(Q, cell, c, beta, D, False, noalloc), want) ** 2).mean()) for noalloc in (False, True)]
    assert rms[0] <= 2 ** 0.5 * rms[1], rms
