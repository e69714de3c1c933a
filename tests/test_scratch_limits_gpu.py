"""The FP64 products' scratch at its limit: the largest allocation of a call, which the digit products' scratch
is, fails once, and the call still succeeds with less.  The failure is a host-side one: a small library,
preloaded into a child process, lets allocations of a given size and above return cudaErrorMemoryAllocation.

Bars: FP64 results of the two runs within 1e-12 of each other's norm (both have FP64 accuracy by norm, the
Davidson's Ritz values after three steps of a converging iteration too), FP32 ones within 1e-6."""
import os
import shutil
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdlib.h>
static size_t limit = (size_t)-1, largest;
static void* real(const char* name) {
    void* h = dlopen("libcudart.so.13", RTLD_NOW | RTLD_NOLOAD);
    return h ? dlsym(h, name) : NULL;
}
static int refuse(size_t n) {
    if (n > largest) largest = n;
    return n >= limit;
}
void fake_limit(size_t n) {
    limit = n;
    largest = 0;
}
size_t fake_largest(void) { return largest; }
int cudaMalloc(void** p, size_t n) {
    int (*f)(void**, size_t) = (int (*)(void**, size_t))real("cudaMalloc");
    return !f || refuse(n) ? 2 : f(p, n);
}
int cudaMallocAsync(void** p, size_t n, void* s) {
    int (*f)(void**, size_t, void*) = (int (*)(void**, size_t, void*))real("cudaMallocAsync");
    return !f || refuse(n) ? 2 : f(p, n, s);
}
"""

CHILD = r"""
import ctypes, sys
import numpy as np, torch
sys.path[:0] = [sys.argv[1], sys.argv[1] + "/tests"]
import qm_synth as S
import paper_2308_07277_gb300 as Q
from cases import make_case
fake = ctypes.CDLL(None)
fake.fake_limit.argtypes, fake.fake_largest.restype = [ctypes.c_size_t], ctypes.c_size_t
d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
rng = np.random.default_rng(1)
z = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
cell = S.cubic_si8(12.0, nbnd=64, reps=(2, 2, 2), kpts=[[0.25, 0.25, 0.25]])
c = make_case(cell, 0)
v, beta, D = (d(c[k]) for k in ("v", "beta", "D"))
A, B = d(z(480, 9000)), d(z(157, 9000))
U = d(np.linalg.qr(z(c["psi"].shape[1], 320))[0].T)
eps, hd, lam = (torch.linspace(0.1, 1.0, n, dtype=torch.float64, device="cuda") for n in (64, U.shape[1], 320))

def call(kind):
    g = Q.qm_gspace_create(cell.lattice, cell.kpts, cell.ecut_ha, cell.grid)
    psi = d(c["psi"])
    try:
        if kind == "zgemm":
            out = Q.qm_zgemm("cn", A, B)
        elif kind == "hpsi":
            out = torch.empty_like(psi)
            for _ in range(2):
                Q.qm_hpsi(g, 0, psi, v, beta, D, out=out)
        elif kind == "davidson":
            return Q.qm_davidson(g, 0, psi, v, beta, D, tol=1e-9, max_iter=3, raise_not_converged=False)[0]
        else:
            out = Q.qm_mlp_pairs(g, 0, psi, psi.flip(0).contiguous(), eps, hd, U, lam, 1e-3)[2]
        torch.cuda.synchronize()
        return out.cpu().numpy()
    finally:
        Q.qm_gspace_destroy(g)

for kind in ("zgemm", "hpsi", "davidson", "pairs"):
    call(kind)                                 # (torch's own blocks are there)
    fake.fake_limit(2 ** 64 - 1)
    full = call(kind)
    n = fake.fake_largest()
    assert n > 70 << 20, (kind, n)             # the digit products' scratch
    fake.fake_limit(n)
    less = call(kind)
    assert fake.fake_largest() == n            # asked for and refused
    fake.fake_limit(2 ** 64 - 1)
    err = np.linalg.norm(less - full) / np.linalg.norm(full)
    print(kind, n, err)
    assert err <= (1e-6 if kind == "pairs" else 1e-12), (kind, err)
"""


def test_less_scratch(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cc = shutil.which("gcc")
    if not cc:
        pytest.skip("no C compiler")
    (tmp_path / "fake.c").write_text(FAKE)
    (tmp_path / "child.py").write_text(CHILD)
    so = str(tmp_path / "fake.so")
    subprocess.run([cc, "-shared", "-fPIC", "-O1", "-o", so, str(tmp_path / "fake.c"), "-ldl"], check=True)
    r = subprocess.run([sys.executable, str(tmp_path / "child.py"), ROOT], env=dict(os.environ, LD_PRELOAD=so), capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr[-3000:]
