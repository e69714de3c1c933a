"""H psi of the precision form under stream capture: the nonlocal chain on the handle's second stream
(its kernels launched while the one before drains) becomes part of the graph, and a replay on other
states gives the call's own result bit for bit.  Sizes: the projection on the CUDA cores, rows that
find their scale in the splitting kernel, sums of the K splits taken in the expansion or on their own."""
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


def dev(a, dt):
    return torch.from_numpy(np.ascontiguousarray(a)).to(dt).cuda()


@pytest.mark.parametrize("reps,nb,prepared", [((1, 1, 1), 4, False), ((1, 1, 1), 64, True), ((2, 2, 1), 3, True),
                                              ((2, 2, 2), 2, True), ((2, 2, 2), 40, False)])
def test_replay_equals_call(Q, reps, nb, prepared):
    cell = S.cubic_si8(15.0, nbnd=nb, reps=reps, kpts=[[0.25, 0.25, 0.25]])
    c = make_case(cell, 0)
    g = Q.qm_gspace_create(cell.lattice, cell.kpts, cell.ecut_ha, cell.grid)
    try:
        psi = [dev(c["psi"], torch.complex64), dev(c["psi"][::-1].copy(), torch.complex64)]
        v, beta, D = dev(c["v"], torch.float64), dev(c["beta"], torch.complex64), dev(c["D"], torch.float64)
        if prepared:
            Q.qm_hpsi_prepare(g, 0, beta)
        want = [Q.qm_hpsi(g, 0, p, v, beta, D, prec="mixed").clone() for p in psi]
        x, out = torch.empty_like(psi[0]), torch.empty_like(psi[0])
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            Q.qm_hpsi(g, 0, x, v, beta, D, out=out, prec="mixed", stream=torch.cuda.current_stream())
        for p, w in list(zip(psi, want)) * 2:
            x.copy_(p)
            out.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(out, w)
    finally:
        Q.qm_gspace_destroy(g)
