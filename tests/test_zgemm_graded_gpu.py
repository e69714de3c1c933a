"""FP64 products whose rows are graded against each other: arith 3 (multiply-adds at every size) keeps FP64
accuracy element by element, arith 0 the bound by norm that qm.h states; and fp64_exact = 1 runs a Davidson
without digit products.

Bars.  arith 3: 1e-14 of sum_k |a_k| |b_k| (random rounding of up to 4000 terms, 1.1e-16 x 8, and the host's
own).  arith 0: every real product's operands are off by at most 2^-55 of their row's largest component and
the dropped digits by 2^-59.7 of both, an output has 2 K real products per component, and is rounded once;
sqrt(2) for the modulus, and the host's own error beside it."""
import ctypes

import numpy as np
import pytest

import qm_synth as S

from cases import make_case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2308_07277_gb300 as Q
    return Q


def _graded(kind, M, N, K):
    rng = np.random.default_rng(M + K)
    z = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    a, b, x = z(M, K), z(N, K), np.linspace(0, 1, K)
    if kind == "spike":      # one element far above the others, where the other operand holds nothing
        a[:, 7] *= 1e16
        b[:, 7] = 0
    else:
        a *= np.exp(-kind * x)
        b *= np.exp(kind * (x - 1))
    return a, b


@pytest.mark.parametrize("kind", [3, 20, 30, 46, "spike"])
@pytest.mark.parametrize("op", ["cn", "tn"])
def test_graded_rows(Q, op, kind):
    M, N, K = (200, 60, 4000) if op == "cn" else (60, 4000, 200)
    a, b = _graded(kind, M, N, K)
    A, B = (torch.from_numpy(np.ascontiguousarray(x if op == "cn" else x.T)).cuda() for x in (a, b))
    ref, bound = (np.conj(a) if op == "cn" else a) @ b.T, np.abs(a) @ np.abs(b).T
    err = np.abs(Q.qm_zgemm(op, A, B, arith=3).cpu().numpy() - ref)
    assert (err <= 1e-14 * bound).all(), (err / bound).max()
    comp = lambda z: np.maximum(np.abs(z.real), np.abs(z.imag)).max(1)
    one = lambda z: (np.abs(z.real) + np.abs(z.imag)).sum(1)
    ma, mb = comp(a)[:, None], comp(b)[None]
    norm = 2.0 ** -55 * (ma * one(b)[None] + mb * one(a)[:, None]) + 2 * K * 2.0 ** -59.7 * ma * mb
    err = np.abs(Q.qm_zgemm(op, A, B, arith=0).cpu().numpy() - ref)
    assert (err <= 2 ** 0.5 * norm + 1e-14 * bound).all(), (err / norm).max()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_fp64_exact_runs_without_digit_products(Q, prec):
    from paper_2308_07277_gb300 import _lib
    lib = _lib.load()
    split = next(i for i in range(64) if lib.qm_prof_name(i) == b"k_split")
    cell = S.cubic_si8(12.0, nbnd=40, reps=(2, 2, 2), kpts=[[0.25, 0.25, 0.25]])
    c = make_case(cell, 0)
    g = Q.qm_gspace_create(cell.lattice, cell.kpts, cell.ecut_ha, cell.grid)
    launches = {}
    try:
        d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
        for exact in (0, 1):
            assert lib.qm_prof_enable(1) == 0
            # (mixed_switch above every residual: the precision form goes straight to its FP64 phase)
            Q.qm_davidson(g, 0, d(c["psi"]), d(c["v"]), d(c["beta"]), d(c["D"]), tol=1e-9, max_iter=3, prec=prec, fp64_exact=exact,
                          mixed_switch=1e6, raise_not_converged=False)
            ms, n = ctypes.c_double(), ctypes.c_longlong()
            assert lib.qm_prof_read(split, ctypes.byref(ms), ctypes.byref(n)) == 0
            launches[exact] = n.value
    finally:
        lib.qm_prof_enable(0)
        Q.qm_gspace_destroy(g)
    # the precision form's FP32 phase has splits of its own, the same number in both calls
    assert launches[1] < launches[0] and (prec == "mixed" or launches[1] == 0), launches
