"""The eigensolver over the range of FP64: matrices scaled far from one and columns whose norm is far
below the matrix's, at sizes of the single-CTA reduction (m <= 64) and just above it, against LAPACK.
Tolerances of the general sizes on the matrix's own scale: 1e-12 |A| for eigenvalues and residuals
(Householder reduction: a few eps per column), 1e-10 for orthonormality.  A coupling below eps |A|
changes nothing at that tolerance, so dropping it is within it too."""
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


def _check(Q, H, nev):
    ev, Y = Q.qm_eigh_lowest(torch.from_numpy(H).cuda(), nev)
    torch.cuda.synchronize()
    ev, Y = ev.cpu().numpy(), Y.cpu().numpy()
    full = np.linalg.eigvalsh(H)
    scale = np.abs(full).max()
    assert np.abs(ev - full[:nev]).max() <= 1e-12 * scale
    assert np.abs(H / scale @ Y - Y * (ev / scale)).max() <= 1e-12
    assert np.abs(Y.conj().T @ Y - np.eye(nev)).max() <= 1e-10


@pytest.mark.parametrize("m", [2, 3, 8, 33, 64, 65])
@pytest.mark.parametrize("power", [-140, -100, -78, -50, -15, 15, 50, 78, 100, 140])
def test_scaled(Q, m, power):
    rng = np.random.default_rng(m)
    X = rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m))
    _check(Q, 10.0 ** power * 0.5 * (X + X.conj().T), m)


@pytest.mark.parametrize("scale", [1.0, 1e90, 1e-90])
@pytest.mark.parametrize("eps", [1e-30, 1e-37, 1e-80, 1e-90, 1e-100, 1e-156])
def test_one_tiny_complex_coupling(Q, eps, scale):
    """A reflector of a column that holds next to nothing."""
    H = np.diag(np.arange(1.0, 9.0)).astype(complex)
    H[1, 0], H[0, 1] = eps * 1j, -eps * 1j
    H[5, 2], H[2, 5] = eps * (1 + 2j), eps * (1 - 2j)
    _check(Q, scale * H, 8)


@pytest.mark.parametrize("m", [6, 40])
def test_graded_columns(Q, m):
    """Rows and columns falling by 300 decades over the matrix."""
    rng = np.random.default_rng(m)
    X = rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m))
    f = 10.0 ** -np.linspace(0, 150, m)
    H = 0.5 * (X + X.conj().T) * f[:, None] * f[None, :]
    _check(Q, H, m)
    _check(Q, np.ascontiguousarray(H[::-1, ::-1]), m)
