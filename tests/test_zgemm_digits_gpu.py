"""The FP64 products on the tensor cores (digit splitting, csrc/zdigits.cu) against a host FP64 product,
at the edges of their tiles (128 x 32 complex outputs, 8 terms per K tile, 128 terms between drains,
K panels) and for rows they leave to the FP64 kernels.

Bar: 1e-14 of sum_k |a_mk| |b_nk| per output.  An operand element is rounded at 2^-55 of its row's
largest component, so a term's error is at most 2^-55 (max|a| |b| + max|b| |a|) per real product and
the sum's at most 2^-52 (max/mean)/K-average: with the largest element at most 20 times the mean
magnitude of its row (normal numbers under a mild decay) that is below 4.5e-15 of the bound, and the
host's own FP64 sum is within 5e-15 of it (random rounding over up to 3e4 terms).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-14


@pytest.fixture(scope="module")
def Q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2308_07277_gb300 as Q
    return Q


def crandn(rng, *shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# the smallest products served are 1.25e7 complex multiply-adds
CN = [(128, 32, 3072), (129, 33, 3001), (127, 31, 3201), (1, 40, 320001), (640, 1, 20001), (300, 299, 1031), (480, 157, 9000),
      (1100, 700, 2500)]
TN = [(32, 12288, 32), (33, 12289, 37), (31, 12287, 33), (1, 200001, 63), (160, 5003, 17), (157, 641, 480), (288, 3000, 1020)]


@pytest.mark.parametrize("M,N,K", CN)
def test_cn(Q, M, N, K):
    rng = np.random.default_rng(M + N + K)
    A = crandn(rng, M, K) * np.exp(-np.linspace(0, 2, K))[None, :]
    B = crandn(rng, N, K) * np.exp(-np.linspace(1, 0, K))[None, :] * 10.0 ** rng.uniform(-3, 3, (N, 1))
    C = Q.qm_zgemm("cn", dev(A), dev(B)).cpu().numpy()
    err = np.abs(C - np.conj(A) @ B.T) / (np.abs(A) @ np.abs(B).T)
    assert err.max() <= TOL, err.max()


@pytest.mark.parametrize("M,N,K", TN)
def test_tn(Q, M, N, K):
    rng = np.random.default_rng(7 * M + N + K)
    A = crandn(rng, K, M) * 10.0 ** rng.uniform(-3, 3, (1, M))
    B = crandn(rng, K, N)
    C = Q.qm_zgemm("tn", dev(A), dev(B)).cpu().numpy()
    err = np.abs(C - A.T @ B) / (np.abs(A).T @ np.abs(B))
    assert err.max() <= TOL, err.max()


@pytest.mark.parametrize("op", ["cn", "tn"])
def test_same_sum_whatever_the_split(Q, op):
    """The integer sums are exact: a row of a product does not depend on the other rows' number
    (which changes splits and panels), bit by bit."""
    rng = np.random.default_rng(5)
    M, N, K = (200, 90, 6001) if op == "cn" else (90, 6001, 200)
    A = crandn(rng, M, K) if op == "cn" else crandn(rng, K, M)
    B = crandn(rng, N, K) if op == "cn" else crandn(rng, K, N)
    full = Q.qm_zgemm(op, dev(A), dev(B)).cpu().numpy()
    part = Q.qm_zgemm(op, dev(A[:45] if op == "cn" else A[:, :45]), dev(B)).cpu().numpy()
    np.testing.assert_array_equal(full[:45], part)


@pytest.mark.parametrize("op", ["cn", "tn"])
def test_rows_left_to_fp64(Q, op):
    """Rows with NaN, infinities, values below 2^-960 and rows of zeros; rows at 1e+-150."""
    rng = np.random.default_rng(9)
    M, N, K = (150, 70, 2000) if op == "cn" else (70, 2000, 150)
    a = crandn(rng, M, K)
    b = crandn(rng, N, K)
    a[3, 5], a[66, 7] = np.nan, np.inf
    a[10] *= 1e-300
    a[11] = 0
    a[12] *= 1e150
    a[13] *= 1e-150
    b[1, 1] = complex(0, -np.inf)
    b[60] *= 1e-150
    with np.errstate(all="ignore"):
        if op == "cn":
            C, ref = Q.qm_zgemm("cn", dev(a), dev(b)), np.conj(a) @ b.T
        else:
            C, ref = Q.qm_zgemm("tn", dev(a.T), dev(b.T)), a @ b.T
        C = C.cpu().numpy()
        bound = np.abs(a) @ np.abs(b).T
    fin = np.isfinite(bound)
    assert fin.sum() == (M - 2) * (N - 1)
    assert not np.isfinite(C[~fin]).any()
    err = np.abs(C - ref)[fin]
    assert np.all(err <= TOL * bound[fin] + 5e-324), (err / np.maximum(bound[fin], 1e-320)).max()
