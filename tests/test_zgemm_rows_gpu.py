"""FP64 products of very many output rows: more than a launch's 65535 row blocks of either kernel (8 rows a
block for cn, 4 or 8 for tn), against a host product.  Bar: 1e-14 of sum_k |a_mk| |b_nk| (three terms: four
roundings of 1.1e-16 and the host's own)."""
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


@pytest.mark.parametrize("op,M", [("cn", 65535 * 8), ("cn", 65535 * 8 + 1), ("tn", 65535 * 4), ("tn", 65535 * 4 + 1),
                                  ("tn", 65535 * 8 + 5)])
def test_many_rows(Q, op, M):
    rng = np.random.default_rng(M)
    N, K = 2, 3
    z = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    a, b = z(M, K), z(N, K)
    A, B = (a, b) if op == "cn" else (a.T, b.T)
    C = Q.qm_zgemm(op, *(torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (A, B))).cpu().numpy()
    ref = (np.conj(a) if op == "cn" else a) @ b.T
    assert (np.abs(C - ref) <= 1e-14 * (np.abs(a) @ np.abs(b).T)).all()


def test_many_rows_split_over_k(Q):
    """The same with partial sums over K (one tile row of columns, K long enough to split)."""
    rng = np.random.default_rng(1)
    z = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    a, b = z(65535 * 8 + 9, 40), z(1, 40)
    C = Q.qm_zgemm("cn", torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()).cpu().numpy()
    assert (np.abs(C - np.conj(a) @ b.T) <= 1e-14 * (np.abs(a) @ np.abs(b).T)).all()
