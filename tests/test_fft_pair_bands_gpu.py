"""The paired FP32 FFT path of H psi (csrc/fft_pair.cuh) with enough transforms that it is taken: every
length it serves on every axis, an odd last band, and at Gamma 1 to 4 bands in the last pair of transforms.

The rule for taking it (pair_path in fft_pair.cu): all three lengths in the list, the plane within 226 KB of
shared memory, and at least two plane blocks per SM; each test asserts it for its own call.  Bars: those of
the precision form (1e-6 per band, 5e-6 element-wise of the band's largest element): FP32 round-off 6e-8
growing with the root of the number of butterfly stages (at most about 30), 3e-7, under a factor of three.
"""
import numpy as np
import pytest

import qm_synth as S
from qm_synth.cells import fcc_lattice
from oracle import gspace as OG
from oracle import hamiltonian as OH

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LENGTHS = [18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 81, 90, 96, 100, 120, 128, 144]
# each length on each axis once; long y beside short z (the plane must fit shared memory)
GRIDS = [(n, LENGTHS[(i + 8) % 25], LENGTHS[24 - (i + 8) % 25]) for i, n in enumerate(LENGTHS)]


@pytest.fixture(scope="module")
def Q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2308_07277_gb300 as Q
    return Q


def pairs_needed(grid):
    """Pairs of transforms from which the grid takes the paired path."""
    assert all(n in LENGTHS for n in grid)
    assert (grid[2] * (grid[1] + 1) + grid[1] + grid[2]) * 16 <= 226 * 1024
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return -(-2 * sms // grid[0])


def dev(a, dtype=None):
    t = torch.from_numpy(np.ascontiguousarray(a))
    return (t if dtype is None else t.to(dtype)).cuda()


def check(got, want):
    got = got.cpu().numpy().astype(np.complex128)
    rel = np.linalg.norm(got - want, axis=1) / np.linalg.norm(want, axis=1)
    el = np.abs(got - want).max(axis=1) / np.abs(want).max(axis=1)
    assert rel.max() <= 1e-6 and el.max() <= 5e-6, (rel.max(), el.max())


@pytest.mark.parametrize("grid", GRIDS, ids=str)
def test_lengths_odd_bands(Q, grid):
    """A small sphere of a skew cell on a large grid, and a sphere that reaches a tenth of each axis."""
    k, nb = (0.25, -0.25, 0.25), 2 * pairs_needed(grid) - 1
    for lat in (fcc_lattice(6.0), np.diag(0.25 * np.asarray(grid))):
        gs = OG.gsphere(lat, grid, 3.0, k)
        g = Q.GSpace(lat, [k], 3.0, grid)
        v = np.random.default_rng(1).standard_normal(int(np.prod(grid)))
        psi = S.psi_random(2, nb, len(gs["idx"]))
        out = g.hpsi(0, dev(psi, torch.complex64), dev(v), None, None, prec="mixed")
        check(out, OH.hpsi_fft(psi, gs, v, None, None))
        g.close()


@pytest.mark.parametrize("last", [1, 2, 3, 4])
@pytest.mark.parametrize("grid", GRIDS[::3] + [GRIDS[22], GRIDS[23]], ids=str)
def test_gamma_bands(Q, grid, last):
    nb = 4 * (pairs_needed(grid) - 1) + last
    lat = np.diag(0.25 * np.asarray(grid))
    gs = OG.gsphere(lat, grid, 3.0)
    g = Q.GSpace(lat, [(0.0, 0.0, 0.0)], 3.0, grid)
    v = np.random.default_rng(1).standard_normal(int(np.prod(grid)))
    psi = S.psi_random_real(3, nb, gs["miller"])
    out = Q.qm_hpsi_gamma(g.handle, 0, dev(psi, torch.complex64), dev(v), None, None, prec="mixed")
    check(out, OH.hpsi_fft(psi, gs, v, None, None))
    g.close()
