"""The precision form's FFT path on two transforms at once (csrc/fft_pair.cuh): every length it serves on
every axis, odd band counts, the Gamma form and GW products, against the oracle; and the grids it leaves to
the single-transform kernels.

Bars: those of the precision form (1e-6 per band, 5e-6 element-wise of the band's largest element): FP32
round-off 6e-8 growing with the root of the number of butterfly stages (at most about 30 over both
transforms of three axes), 3e-7, under a factor of three of margin.
"""
import numpy as np
import pytest

import qm_synth as S
from qm_synth.cells import fcc_lattice
from oracle import gspace as OG
from oracle import gw as OW
from oracle import hamiltonian as OH

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LENGTHS = [18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 81, 90, 96, 100, 120, 128, 144]
# each length on each axis once; long y beside short z (two planes fit shared memory)
GRIDS = [(n, LENGTHS[(i + 8) % 25], LENGTHS[24 - (i + 8) % 25]) for i, n in enumerate(LENGTHS)]
SINGLE = [(16, 18, 18), (24, 125, 27), (108, 20, 20), (20, 144, 128), (135, 15, 10)]   # lengths or planes not served


@pytest.fixture(scope="module")
def Q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2308_07277_gb300 as Q
    return Q


def dev(a, dtype=None):
    t = torch.from_numpy(np.ascontiguousarray(a))
    return (t if dtype is None else t.to(dtype)).cuda()


def check(got, want):
    got = got.cpu().numpy().astype(np.complex128)
    rel = np.linalg.norm(got - want, axis=1) / np.linalg.norm(want, axis=1)
    el = np.abs(got - want).max(axis=1) / np.abs(want).max(axis=1)
    assert rel.max() <= 1e-6 and el.max() <= 5e-6, (rel.max(), el.max())


@pytest.mark.parametrize("grid", GRIDS + SINGLE, ids=str)
def test_lengths(Q, grid):
    """A small sphere of a skew cell on a large grid, and a sphere that reaches a tenth of each axis."""
    k = (0.25, -0.25, 0.25)
    for lat in (fcc_lattice(6.0), np.diag(0.25 * np.asarray(grid))):
        gs = OG.gsphere(lat, grid, 3.0, k)
        g = Q.GSpace(lat, [k], 3.0, grid)
        assert np.array_equal(g.indices(0)[0], gs["idx"])
        v = np.random.default_rng(1).standard_normal(int(np.prod(grid)))
        psi = S.psi_random(2, 3, len(gs["idx"]))
        out = g.hpsi(0, dev(psi, torch.complex64), dev(v), None, None, prec="mixed")
        check(out, OH.hpsi_fft(psi, gs, v, None, None))
        g.close()


@pytest.mark.parametrize("nb", [1, 2, 3, 4, 5, 7])
def test_gamma_band_counts(Q, nb):
    cell = S.cubic_si8(10.0, nbnd=6)
    grid = OG.fft_grid(cell.lattice, 4 * cell.ecut_ha)
    gs = OG.gsphere(cell.lattice, grid, cell.ecut_ha, cell.kpts[0])
    v = S.vloc_on_grid(cell.lattice, cell.tau, grid)
    psi = S.psi_random_real(3, nb, gs["miller"])
    g = Q.GSpace(cell.lattice, cell.kpts, cell.ecut_ha, grid)
    out = Q.qm_hpsi_gamma(g.handle, 0, dev(psi, torch.complex64), dev(v), None, None, prec="mixed")
    check(out, OH.hpsi_fft(psi, gs, v, None, None))
    g.close()


@pytest.mark.parametrize("nl,nr", [(1, 1), (2, 3), (3, 4)])
def test_gw_state_counts(Q, nl, nr):
    cell = S.fcc_si2(16.0, kpts=[[0.25, -0.25, 0.25], [0.0, 0.0, 0.0]])
    grid = OG.fft_grid(cell.lattice, 4 * cell.ecut_ha)
    sl, sr = (OG.gsphere(cell.lattice, grid, cell.ecut_ha, k) for k in cell.kpts)
    q = cell.kpts[0] - cell.kpts[1]
    se = OG.gsphere(cell.lattice, grid, 0.5 * cell.ecut_ha, q)
    g, ge = Q.GSpace(cell.lattice, cell.kpts, cell.ecut_ha, grid), Q.GSpace(cell.lattice, [q], 0.5 * cell.ecut_ha, grid)
    pl, pr = S.psi_random(1, nl, len(sl["idx"])), S.psi_random(2, nr, len(sr["idx"]))
    M = Q.qm_gw_mel(g.handle, 0, 1, dev(pl, torch.complex64), dev(pr, torch.complex64), ge.handle, 0, len(se["idx"]), prec="mixed")
    check(M, OW.mel_fft(pl, sl, pr, sr, se))
    ge.close()
    g.close()
