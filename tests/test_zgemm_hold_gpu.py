"""FP64 products in several panels of digit planes: the same result whatever the scratch, and bounded waits
that run out in one panel (qm_zgemm_hold: no polls at all, so every block of that panel gives up at once and
drains its own copies) leave no incomplete sum behind: the rows are recomputed in FP64 multiply-adds.
Bar: 1e-14 of sum_k |a_mk| |b_nk| (operands rounded at 2^-55 of the row's largest, at most 5 times its mean)."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2308_07277_gb300  # noqa: F401
    from paper_2308_07277_gb300 import _lib
    return _lib.load()


def _product(lib, op, A, B, M, N, K, scratch, panel=-1, polls=0):
    C = torch.full((M, N), complex("nan"), dtype=torch.complex128, device="cuda")
    n = ctypes.c_int(-1)
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    st = lib.qm_zgemm_hold(op, M, N, K, p(A), A.stride(0), p(B), B.stride(0), p(C), N, scratch, panel, polls, ctypes.byref(n),
                           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    return C.cpu().numpy(), n.value


# (scratch for the whole product, for several panels)
@pytest.mark.parametrize("op,M,N,K,scratch", [(0, 150, 40, 8001, 24 << 20), (1, 40, 8001, 150, 9 << 20)])
def test_expired_panel(lib, op, M, N, K, scratch):
    rng = np.random.default_rng(M)
    z = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    a, b = z(M, K), z(N, K)
    ref, bound = (np.conj(a) if op == 0 else a) @ b.T, np.abs(a) @ np.abs(b).T
    A, B = (torch.from_numpy(np.ascontiguousarray(x if op == 0 else x.T)).cuda() for x in (a, b))
    whole, n1 = _product(lib, op, A, B, M, N, K, 1 << 29)
    parts, n = _product(lib, op, A, B, M, N, K, scratch)
    assert n1 == 1 and n >= 3, (n1, n)
    assert (np.abs(whole - ref) <= 1e-14 * bound).all()
    np.testing.assert_array_equal(parts, whole)      # the sums are exact integers
    for panel in range(n):
        C, _ = _product(lib, op, A, B, M, N, K, scratch, panel)
        assert (np.abs(C - ref) <= 1e-14 * bound).all(), panel
    none, n0 = _product(lib, op, A, B, M, N, K, 0)
    assert n0 == 0 and (np.abs(none - ref) <= 1e-14 * bound).all()
