"""The eigensolver's single-CTA reduction (m <= 64) at the edges of its warps and of its range, the
Sturm counts at extreme scales and with decoupled or exactly repeated diagonals, and the inverse
iteration past the shared memory of resident blocks, against LAPACK.  Tolerances as for the general
sizes, on the matrix's own scale: 1e-12 |A| for eigenvalues and eigen-residuals (Householder
reduction: a few eps per column, 64 x 3.3e-16 x 10), 1e-10 for orthonormality (eps |T| / gap outside
the clusters that are orthogonalised)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2308_07277_gb300 as Q
    return Q


def _herm(rng, m):
    X = rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m))
    return 0.5 * (X + X.conj().T)


def _check(Q, H, nev):
    ev, Y = Q.qm_eigh_lowest(torch.from_numpy(H).cuda(), nev)
    torch.cuda.synchronize()
    ev, Y = ev.cpu().numpy(), Y.cpu().numpy()
    full = np.linalg.eigvalsh(H)
    scale = np.abs(full).max()
    assert np.abs(ev - full[:nev]).max() <= 1e-12 * scale
    assert np.abs(H @ Y - Y * ev).max() <= 1e-12 * scale
    assert np.abs(Y.conj().T @ Y - np.eye(nev)).max() <= 1e-10


@pytest.mark.parametrize("m", [2, 4, 9, 16, 31, 32, 33, 63, 64, 65])
@pytest.mark.parametrize("scale", [1.0, 1e-60, 1e60])
def test_random(Q, m, scale):
    _check(Q, scale * _herm(np.random.default_rng(m), m), m)


@pytest.mark.parametrize("m", [8, 40, 64])
def test_repeated_diagonal(Q, m):
    _check(Q, 0.7 * np.eye(m, dtype=complex), m)
    d = np.repeat([1.0, -2.0, 3.0, 0.0], m // 4)
    _check(Q, np.diag(d).astype(complex), m)


@pytest.mark.parametrize("m", [24, 64, 90])
def test_decoupled_tridiagonal(Q, m):
    """Couplings from 1 down to 1e-30 beside equal diagonal entries."""
    e = 10.0 ** -np.linspace(0, 30, m - 1)
    H = np.diag(np.tile([1.0, 1.0, -1.0, 0.25], m)[:m]) + np.diag(e, 1) + np.diag(e, -1)
    _check(Q, H.astype(complex), m)


@pytest.mark.parametrize("m", [66, 127, 128, 129, 256, 257, 512, 513, 768, 769])
def test_back_transformation_rows(Q, m):
    """The register rows of the back-transformation at their edges, with reflectors that are the identity
    (a block that is already diagonal) between the others."""
    H = _herm(np.random.default_rng(m), m)
    H[m // 3: m // 2, :] = 0.0
    H[:, m // 3: m // 2] = 0.0
    H[np.arange(m // 3, m // 2), np.arange(m // 3, m // 2)] = 200.0 + np.arange(m // 2 - m // 3)
    _check(Q, H, 9)


def test_inverse_iteration_past_shared_memory(Q):
    _check(Q, _herm(np.random.default_rng(3), 1216), 470)
