"""The work a user of the library has it do, as cases that can be timed: H psi in both precisions
(smallest, ordinary and largest cell), its Gamma form, the batched plan, the Davidson's
plane-wave-length products, a self-consistency run, a real-time step, GW matrix elements and the
learned preconditioner's training gradient.

Cells are diamond-silicon supercells (fcc or cubic, n1 x n2 x n3 repetitions, a0 = 10.26 bohr) with
Gaussian local wells and Gaussian s + p projectors, the workloads of bench.py and the tests; the
seed displaces the atoms by up to 1 % of a0 per component and draws the states: complex normal
coefficients, the starting states of bench.py and the tests.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2308_07277_gb300 as Q

A0 = 10.26
DEPTH, RC = -1.5, 1.0
D_ATOM = (5.0, 1.5, 1.5, 1.5)
SITES8 = ((0, 0, 0), (0, .5, .5), (.5, 0, .5), (.5, .5, 0),
          (.25, .25, .25), (.25, .75, .75), (.75, .25, .75), (.75, .75, .25))
MP4 = ((.25, .25, .25), (.25, .25, -.25), (.25, -.25, .25), (-.25, .25, .25))


# ------------------------------------------------------------------ cells and inputs
def _geometry(kind, reps):
    """Lattice rows and ideal atom sites (bohr)."""
    reps = np.asarray(reps)
    if kind == "fcc":
        prim = 0.5 * A0 * np.array([[-1., 0, 1], [0, 1, 1], [-1, 1, 0]])
        basis = np.array([[0., 0, 0], [.25 * A0] * 3])
    else:
        prim = A0 * np.eye(3)
        basis = A0 * np.array(SITES8, float)
    n = np.stack(np.meshgrid(*[np.arange(r) for r in reps], indexing="ij"), -1).reshape(-1, 3)
    return prim * reps[:, None], (basis[None] + (n @ prim)[:, None]).reshape(-1, 3)


def _natoms(case):
    return (2 if case["kind"] == "fcc" else 8) * case["r1"] * case["r2"] * case["r3"] - case.get("vacancy", 0)


def _npw(case, ecut_ry=None):
    """Plane waves of the sphere, from its volume (work estimates)."""
    vol = abs(np.linalg.det(_geometry(case["kind"], (case["r1"], case["r2"], case["r3"]))[0]))
    return vol * (case["ecut_ry"] if ecut_ry is None else ecut_ry) ** 1.5 / (6 * math.pi ** 2)


def _nr(case):
    """Grid points by the grid rule (or the stated grid)."""
    if case.get("g1"):
        return case["g1"] * case["g2"] * case["g3"]
    lat = _geometry(case["kind"], (case["r1"], case["r2"], case["r3"]))[0]
    return float(np.prod([_grid_n(np.linalg.norm(a), case["ecut_ry"]) for a in lat]))


def _grid_n(length, ecut_ry):
    n = 2 * int(math.sqrt(4 * ecut_ry) * length / (2 * math.pi)) + 1
    while True:
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            return n
        n += 1


class _Cell:
    """A displaced supercell on the GPU: handle, potential, projectors and random states."""

    def __init__(self, case, kpts, gen):
        lat, tau = _geometry(case["kind"], (case["r1"], case["r2"], case["r3"]))
        tau = torch.from_numpy(tau[case.get("vacancy", 0):]).cuda()
        self.tau = tau + (torch.rand(tau.shape, generator=gen, device="cuda", dtype=torch.float64) * 2 - 1) * 0.01 * A0
        self.lat, self.omega = lat, abs(float(np.linalg.det(lat)))
        grid = (case["g1"], case["g2"], case["g3"]) if case.get("g1") else None
        self.ecut = 0.5 * case["ecut_ry"]
        self.g = Q.GSpace(lat, kpts, self.ecut, grid)
        self.D = torch.tensor(D_ATOM, dtype=torch.float64, device="cuda").repeat(len(tau))
        self.vloc = self._potential()

    def _potential(self):
        """Sum of Gaussian wells of width 1 bohr, from its Fourier coefficients."""
        grid = self.g.grid
        recip = 2 * math.pi * np.linalg.inv(self.lat).T
        m = np.stack(np.meshgrid(*[np.fft.fftfreq(n, 1 / n) for n in grid], indexing="ij"), -1)
        G = torch.from_numpy(m.transpose(2, 1, 0, 3).reshape(-1, 3) @ recip).cuda()
        damp = DEPTH * (2 * math.pi) ** 1.5 / self.omega * torch.exp(-0.5 * (G * G).sum(1))
        s = torch.zeros(len(G), dtype=torch.complex128, device="cuda")
        for t in self.tau.split(16):
            ph = G @ t.T
            s += torch.complex(torch.cos(ph), -torch.sin(ph)).sum(1)
        v = torch.fft.ifftn((damp * s).reshape(grid[::-1])).real * float(np.prod(grid))
        return v.reshape(-1).contiguous()

    def sphere(self, ik):
        idx, mil, kpg = self.g.indices(ik)
        return torch.from_numpy(idx).long().cuda(), mil, torch.from_numpy(kpg).cuda()

    def beta(self, q, dtype):
        """Unit-norm Gaussian s and p projectors (4 per atom, npw) at the wavevectors q."""
        g = torch.exp(-0.5 * RC * RC * (q * q).sum(1)) / math.sqrt(self.omega)
        out = torch.empty((4 * len(self.tau), len(q)), dtype=dtype, device="cuda")
        cs, cp = 2 ** 1.5 * math.pi ** .75 * RC ** 1.5, 4 * math.pi ** .75 * RC ** 2.5
        for a, t in enumerate(self.tau):
            ph = q @ t
            e = torch.complex(torch.cos(ph), -torch.sin(ph)) * g
            out[4 * a] = cs * e
            out[4 * a + 1:4 * a + 4] = cp * q.T * e
        return out

    def states(self, nb, q, gen, dtype, mil=None):
        """Complex normal states, normalised per band; real in real space when mil is given."""
        z = torch.randn((nb, len(q), 2), generator=gen, device="cuda", dtype=torch.float64)
        z = torch.view_as_complex(z)
        if mil is not None:
            n = np.asarray(self.g.grid)
            flat = lambda m: ((m % n) * [1, n[0], n[0] * n[1]]).sum(1)
            pos = np.zeros(int(n.prod()), np.int64)
            pos[flat(mil)] = np.arange(len(mil))
            z = z + z[:, torch.from_numpy(pos[flat(-mil)]).cuda()].conj()
        z /= torch.linalg.vector_norm(z, dim=1, keepdim=True)
        return z.to(dtype)


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _ctype(case):
    return torch.complex64 if case["prec"] == "mixed" else torch.complex128


def _kpt(case):
    return [[case["k1"], case["k2"], case["k3"]]]


# ------------------------------------------------------------------ 64-bit references (plain torch)
def _box_fft(psi, idx, grid, inverse=True):
    nr = grid[0] * grid[1] * grid[2]
    box = torch.zeros((len(psi), nr), dtype=torch.complex128, device="cuda")
    box[:, idx] = psi.to(torch.complex128)
    return torch.fft.ifftn(box.reshape((len(psi),) + tuple(grid[::-1])), dim=(1, 2, 3)) * nr


def _h_ref(psi, idx, q, grid, v, beta, D):
    """H psi in 64 bits."""
    psi = psi.to(torch.complex128)
    out = 0.5 * (q * q).sum(1) * psi
    for i in range(0, len(psi), 32):
        u = _box_fft(psi[i:i + 32], idx, grid) * v.reshape(tuple(grid[::-1]))
        out[i:i + 32] += torch.fft.fftn(u, dim=(1, 2, 3)).reshape(len(u), -1)[:, idx] / v.numel()
    if beta is not None:
        b = beta.to(torch.complex128)
        out += ((psi @ b.conj().T) * D) @ b
    return out


# ------------------------------------------------------------------ H psi (and its Gamma form)
def _prep_hpsi(case, seed):
    gen = _gen(seed)
    c = _Cell(case, _kpt(case), gen)
    idx, mil, q = c.sphere(0)
    dt = _ctype(case)
    beta = c.beta(q, dt)
    psi = c.states(case["nb"], q, gen, dt, mil if case["op"] == "gamma" else None)
    if case.get("prepared"):
        Q.qm_hpsi_prepare(c.g.handle, 0, beta)
    return {"case": case, "c": c, "psi": psi, "beta": beta, "out": torch.empty_like(psi), "idx": idx, "q": q}


def _run_hpsi(s):
    f = Q.qm_hpsi_gamma if s["case"]["op"] == "gamma" else Q.qm_hpsi
    return f(s["c"].g.handle, 0, s["psi"], s["c"].vloc, s["beta"], s["c"].D, out=s["out"], prec=s["case"]["prec"])


def _exact_hpsi(s):
    return _h_ref(s["psi"], s["idx"], s["q"], s["c"].g.grid, s["c"].vloc, s["beta"], s["c"].D)


def _work_hpsi(case, nb=None):
    """psi, beta and V read once, the result written once; transforms and projector products."""
    nb = case["nb"] if nb is None else nb
    cs = 8 if case["prec"] == "mixed" else 16
    npw, nr, npj = _npw(case), _nr(case), 4 * _natoms(case)
    fft = nb * (1 if case["op"] != "gamma" else .5) * 5 * nr * math.log2(nr) * 2 * 0.6   # pruned, both ways
    return {"bytes": cs * (2 * nb * npw + npj * npw) + 8 * nr, "flops": 16 * npj * npw * nb + fft}


# ------------------------------------------------------------------ batched plan of uneven cells
BATCH = (("fcc", 1, 1, 1), ("fcc", 2, 1, 1), ("fcc", 2, 2, 1), ("cubic", 1, 1, 1), ("fcc", 2, 2, 2))


def _batch_jobs(case):
    """The uneven cells of a batch: family, cutoff, bands and k-points per cell (by the case's own number)."""
    rng = np.random.default_rng([case["cells_seed"], 3])
    jobs = []
    while len(jobs) < case["ncell"]:
        kind, r1, r2, r3 = BATCH[int(rng.integers(5))]
        sub = {"kind": kind, "r1": r1, "r2": r2, "r3": r3, "ecut_ry": float(rng.uniform(15, 30)), "prec": case["prec"],
               "op": "hpsi", "nb": int(rng.integers(8, 49)), "nk": int(rng.integers(1, 9))}
        lat = _geometry(kind, (r1, r2, r3))[0]
        if all(18 <= _grid_n(np.linalg.norm(a), sub["ecut_ry"]) <= 48 for a in lat):
            jobs.append(sub)
    return jobs


def _prep_batch(case, seed):
    gen, dt, cells, todo, total = _gen(seed), _ctype(case), [], [], 0
    kall = np.array([[a, b, d] for a in (.25, -.25) for b in (.25, -.25) for d in (.25, -.25)])
    for sub in _batch_jobs(case):
        c = _Cell(sub, kall[:sub["nk"]], gen)
        cells.append(c)
        for ik in range(sub["nk"]):
            idx, _, q = c.sphere(ik)
            todo.append((c, ik, idx, q, c.states(sub["nb"], q, gen, dt), c.beta(q, dt), total))
            total += sub["nb"] * len(q)
    out = torch.empty(total, dtype=dt, device="cuda")
    jobs = [{"g": c.g.handle, "ik": ik, "psi": psi, "vloc": c.vloc, "beta": beta, "D": c.D,
             "out": out[o:o + psi.numel()].view(psi.shape)} for c, ik, _, _, psi, beta, o in todo]
    # a launch shape such as the autotuner picks for these cells, so that making the plan is quick
    plan = Q.Batch(jobs, prec=case["prec"], ctas_per_sm=3 if case["prec"] == "mixed" else 1, item_points=8192, group_mb=-1)
    return {"case": case, "plan": plan, "out": out, "todo": todo, "cells": cells}


def _run_batch(s):
    s["plan"].run()
    return s["out"]


def _exact_batch(s):
    return torch.cat([_h_ref(psi, idx, q, c.g.grid, c.vloc, beta, c.D).reshape(-1)
                      for c, _, idx, q, psi, beta, _ in s["todo"]])


def _work_batch(case):
    w = {"bytes": 0.0, "flops": 0.0}
    for sub in _batch_jobs(case):
        x = _work_hpsi(sub)
        w = {k: w[k] + sub["nk"] * x[k] for k in w}
    return w


# ------------------------------------------------------------------ Davidson's plane-wave-length products
def _prep_zgemm(case, seed):
    gen = _gen(seed)
    M, N, K = case["m"], case["n"], case["k"]

    def rows(n, length):   # orthonormal-like rows: unit norm, falling off along the plane waves
        z = torch.view_as_complex(torch.randn((n, length, 2), generator=gen, device="cuda", dtype=torch.float64))
        z = z / (1 + torch.linspace(0, 1, length, device="cuda", dtype=torch.float64) ** (2 / 3) * 12)
        return z / torch.linalg.vector_norm(z, dim=1, keepdim=True)

    if case["product"] == "cn":      # overlaps <V_i | H V_j>
        return {"case": case, "A": rows(M, K), "B": rows(N, K)}
    coef = torch.view_as_complex(torch.randn((K, M, 2), generator=gen, device="cuda", dtype=torch.float64))
    coef = coef * torch.exp(-torch.linspace(0, 8, K, device="cuda", dtype=torch.float64))[:, None]
    coef = (coef / torch.linalg.vector_norm(coef, dim=0, keepdim=True)).contiguous()
    return {"case": case, "A": coef, "B": rows(K, N)}   # rotation to the Ritz vectors


def _run_zgemm(s):
    return Q.qm_zgemm(s["case"]["product"], s["A"], s["B"], arith=s["case"]["arith"])


def _exact_zgemm(s):
    return s["A"].conj() @ s["B"].T if s["case"]["product"] == "cn" else s["A"].T @ s["B"]


def _work_zgemm(case):
    m, n, k = case["m"], case["n"], case["k"]
    return {"bytes": 16.0 * (m * k + n * k + m * n), "flops": 8.0 * m * n * k}


# ------------------------------------------------------------------ real-time propagation
def _prep_etrs(case, seed):
    s = _prep_hpsi(case, seed)
    s["v2"] = s["c"].vloc * (1 + 0.01 * torch.rand((), generator=_gen(seed + 1), device="cuda", dtype=torch.float64))
    s["work"] = torch.empty(2 * s["psi"].numel(), dtype=s["psi"].dtype, device="cuda")
    return s


def _run_etrs(s):
    c, case = s["c"], s["case"]
    return Q.qm_tddft_etrs(c.g.handle, 0, s["psi"], c.vloc, s["v2"], s["beta"], c.D, case["dt"], order=case["order"],
                           prec=case["prec"], work=s["work"])


def _exact_etrs(s):
    case, x = s["case"], s["psi"].to(torch.complex128)
    for v in (s["c"].vloc, s["v2"]):
        u = x
        for r in range(1, case["order"] + 1):
            u = (-0.5j * case["dt"] / r) * _h_ref(u, s["idx"], s["q"], s["c"].g.grid, v, s["beta"], s["c"].D)
            x = x + u
    return x


def _work_etrs(case):
    w = _work_hpsi(case)
    w["flops"] *= 2 * case["order"]
    return w


# ------------------------------------------------------------------ GW matrix elements
def _prep_gw(case, seed):
    gen = _gen(seed)
    kl, kr = np.array(MP4[1]), np.array(MP4[0])
    c = _Cell(case, [kl, kr], gen)
    ge = Q.GSpace(c.lat, [kl - kr], c.ecut * case["eps_frac"], c.g.grid)
    sl, sr = c.sphere(0), c.sphere(1)
    dt = _ctype(case)
    return {"case": case, "c": c, "ge": ge, "sl": sl, "sr": sr, "psil": c.states(case["nl"], sl[2], gen, dt),
            "psir": c.states(case["nr"], sr[2], gen, dt)}


def _run_gw(s):
    return Q.qm_gw_mel(s["c"].g.handle, 0, 1, s["psil"], s["psir"], s["ge"].handle, 0, s["ge"].npw[0], prec=s["case"]["prec"])


def _exact_gw(s):
    grid = s["c"].g.grid
    ul, ur = _box_fft(s["psil"], s["sl"][0], grid), _box_fft(s["psir"], s["sr"][0], grid)
    idx = torch.from_numpy(s["ge"].indices(0)[0]).long().cuda()
    rows = []
    for u in ul:
        for x in ur.split(16):
            f = torch.fft.fftn(u * x.conj(), dim=(1, 2, 3)).reshape(len(x), -1)[:, idx]
            rows.append(f.conj() / float(np.prod(grid)))
    return torch.cat(rows)


def _work_gw(case):
    cs = 8 if case["prec"] == "mixed" else 16
    npw, nr, nq = _npw(case), _nr(case), _npw(case, case["ecut_ry"] * case["eps_frac"])
    pairs, st = case["nl"] * case["nr"], case["nl"] + case["nr"]
    return {"bytes": cs * (st * npw + pairs * nq), "flops": (st * .6 + pairs * .6) * 5 * nr * math.log2(nr) + 6 * pairs * nr}


# ------------------------------------------------------------------ self-consistency (a whole call)
def _prep_scf(case, seed):
    gen = _gen(seed)
    c = _Cell(case, MP4[:case["nk"]], gen)
    sp = [c.sphere(ik) for ik in range(case["nk"])]
    ld = c.g.npw_max
    psis, betas = [], []
    for _, _, q in sp:
        for rows, to in ((c.states(case["nb"], q, gen, torch.complex128), psis), (c.beta(q, torch.complex128), betas)):
            x = torch.zeros((len(rows), ld), dtype=torch.complex128, device="cuda")
            x[:, :len(q)] = rows
            to.append(x)
    return {"case": case, "c": c, "sp": sp, "psis": psis, "betas": betas}


def _run_scf(s):
    case, c = s["case"], s["c"]
    eigs, rho, v, _ = Q.qm_scf(c.g.handle, case["nelec"], [1 / case["nk"]] * case["nk"], [p.clone() for p in s["psis"]],
                               c.vloc, s["betas"], c.D, max_iter=case["steps"], dav_tol=1e-11, prec=case["prec"],
                               raise_not_converged=False)
    return {"eigs": eigs, "rho": rho, "v": v}


def _xc(n):
    """LDA potential: Slater exchange, Perdew-Zunger 1981 correlation, unpolarised."""
    rs = (3 / (4 * math.pi * n.clamp_min(1e-12))) ** (1 / 3)
    sq, lr = rs.sqrt(), rs.log()
    den = 1 + 1.0529 * sq + 0.3334 * rs
    hi = -0.1423 / den * (1 + 7 / 6 * 1.0529 * sq + 4 / 3 * 0.3334 * rs) / den
    lo = 0.0311 * lr + (-0.048 - 0.0311 / 3) + 2 / 3 * 0.002 * rs * lr + (-2 * 0.0116 - 0.002) / 3 * rs
    vx = -(3 / (2 * math.pi)) ** (2 / 3) / rs
    return torch.where(n > 1e-12, vx + torch.where(rs >= 1, hi, lo), torch.zeros_like(n))


def _exact_scf(s):
    """Two steps by dense diagonalisation (linear mixing, as the first mixing step is)."""
    case, c = s["case"], s["c"]
    if case["steps"] > 2 or max(c.g.npw) > 1500:
        return None
    grid = c.g.grid
    nr = c.vloc.numel()
    gr = Q.GSpace(c.lat, [[0, 0, 0]], 4 * c.ecut, grid)
    gidx, _, G = gr.indices(0)
    gidx, g2 = torch.from_numpy(gidx).long().cuda(), (torch.from_numpy(G).cuda() ** 2).sum(1)
    rho = torch.full((nr,), case["nelec"] / c.omega, dtype=torch.float64, device="cuda")
    n = torch.tensor(grid, device="cuda")
    for step in range(case["steps"]):
        ng = torch.fft.fftn(rho.reshape(grid[::-1])).reshape(-1) / nr
        vg = torch.zeros(nr, dtype=torch.complex128, device="cuda")
        vg[gidx] = torch.where(g2 > 1e-9, 4 * math.pi * ng[gidx] / g2.clamp_min(1e-9), torch.zeros_like(ng[gidx]))
        v = c.vloc + (torch.fft.ifftn(vg.reshape(grid[::-1])) * nr).real.reshape(-1) + _xc(rho)
        vt = torch.fft.fftn(v.reshape(grid[::-1])).reshape(-1) / nr
        new, eigs = torch.zeros_like(rho), []
        for (idx, mil, q), b in zip(s["sp"], s["betas"]):
            m = torch.from_numpy(mil).cuda().long()
            d = (m[:, None, :] - m[None, :, :]) % n
            b = b[:, :len(q)]
            H = vt[d[..., 0] + n[0] * (d[..., 1] + n[1] * d[..., 2])] + torch.diag(0.5 * (q * q).sum(1))
            H = H + (b * c.D[:, None]).T @ b.conj()
            w, U = torch.linalg.eigh(H)
            eigs.append(w[:case["nb"]])
            u = _box_fft(U[:, :case["nelec"] // 2].T, idx, grid).reshape(case["nelec"] // 2, -1)
            new += 2 / (case["nk"] * c.omega) * (u.real ** 2 + u.imag ** 2).sum(0)
        if step + 1 < case["steps"]:
            rho = rho + 0.5 * (new - rho)
    return {"eigs": torch.stack(eigs), "rho": rho, "v": v}


def _work_scf(case):
    """About 20 applications of H to every band for each solve (psi, beta and V read once a step)."""
    one = _work_hpsi(case)
    f = case["steps"] * case["nk"]
    return {"bytes": f * one["bytes"], "flops": f * 20.0 * one["flops"]}


# ------------------------------------------------------------------ learned preconditioner, training gradient
def _prep_mlp(case, seed):
    gen = _gen(seed)
    nb, npw = case["bands"], case["npw"]
    n = nb * npw
    rnd = lambda *s: torch.randn(s, generator=gen, device="cuda")
    # kinetic ratio of a sphere (volume element), Ritz value and diagonal in units of the band's kinetic energy
    x = (torch.rand((nb, npw), generator=gen, device="cuda") ** (2 / 3)) * (6 + 2 * rnd(nb, 1).abs())
    e = (0.5 + 0.3 * rnd(nb, 1)).expand(nb, npw)
    f = torch.stack([x, e, x - e + 0.2 * rnd(nb, npw).abs()], -1).reshape(n, 3).contiguous()
    r = torch.view_as_complex(rnd(nb, npw, 2)) / (1 + x)
    dl = -r / (1 + x) + 0.1 * torch.view_as_complex(rnd(nb, npw, 2)) / (1 + x) ** 2
    W1, W2, w3 = rnd(64, 3) / 3 ** .5, rnd(64, 64) / 8, rnd(64) / 8
    z = torch.zeros(64, device="cuda")
    theta = torch.cat([W1.reshape(-1), z, W2.reshape(-1), z, w3, z[:1]])
    w = (r.abs() ** 2).sum(1)
    return {"case": case, "off": torch.arange(nb + 1, device="cuda") * npw, "f": f, "r2": (r.abs() ** 2).reshape(-1),
            "c": (r.conj() * dl).real.reshape(-1).contiguous(), "D": (dl.abs() ** 2).sum(1), "W": w / w.sum(), "theta": theta}


def _run_mlp(s):
    loss, grad = Q.qm_mlp_loss_grad(s["off"], s["f"], s["r2"], s["c"], s["D"], s["theta"], W=s["W"])
    return {"loss": loss, "grad": grad}


def _exact_mlp(s):
    nb, npw = s["case"]["bands"], s["case"]["npw"]
    th = s["theta"].double().requires_grad_(True)
    W1, b1, W2, b2, w3, b3 = (t for t in th.split([192, 64, 4096, 64, 64, 1]))
    D, W = s["D"].double(), s["W"].double()
    loss = 0.0
    for b in range(nb):
        sl = slice(b * npw, (b + 1) * npw)
        f = s["f"][sl].double()
        silu = torch.nn.functional.silu
        h = silu(silu(f @ W1.reshape(64, 3).T + b1) @ W2.reshape(64, 64).T + b2) @ w3 + b3
        x = f[:, 0]
        p = 27 + 18 * x + 12 * x ** 2 + 8 * x ** 3
        K = p / (p + 16 * x ** 4) * torch.nn.functional.softplus(h) / math.log(2)
        A, B = (K * K * s["r2"][sl].double()).sum(), (K * s["c"][sl].double()).sum()
        one = W[b] * (1 - B * B / (A * D[b])) / W.sum()
        one.backward(retain_graph=b + 1 < nb)
        loss += float(one)
    return {"loss": loss, "grad": th.grad}


def _work_mlp(case):
    n = case["bands"] * case["npw"]
    return {"bytes": 20.0 * n, "flops": 6.0 * n * (3 * 64 + 64 * 64 + 64)}


# ------------------------------------------------------------------ the interface
OPS = {"hpsi": (_prep_hpsi, _run_hpsi, _exact_hpsi, _work_hpsi), "gamma": (_prep_hpsi, _run_hpsi, _exact_hpsi, _work_hpsi),
       "batch": (_prep_batch, _run_batch, _exact_batch, _work_batch), "zgemm": (_prep_zgemm, _run_zgemm, _exact_zgemm, _work_zgemm),
       "etrs": (_prep_etrs, _run_etrs, _exact_etrs, _work_etrs), "gw": (_prep_gw, _run_gw, _exact_gw, _work_gw),
       "scf": (_prep_scf, _run_scf, _exact_scf, _work_scf), "mlp": (_prep_mlp, _run_mlp, _exact_mlp, _work_mlp)}


def _cell(kind, r1, r2, r3, ecut_ry, k=(0.0, 0.0, 0.0), **more):
    return {"kind": kind, "r1": r1, "r2": r2, "r3": r3, "ecut_ry": ecut_ry, "k1": k[0], "k2": k[1], "k3": k[2], **more}


def listed():
    cube64 = _cell("cubic", 2, 2, 2, 25.0, MP4[0], g1=72, g2=72, g3=72)
    return [
        # the two-atom cell: one H psi of the smallest Davidson, where launches and latency count
        {"name": "hpsi_si2_fp64", "op": "hpsi", **_cell("fcc", 1, 1, 1, 20.0), "nb": 8, "prec": "fp64"},
        # one k-point of the 64-atom cell in either precision: the ordinary supercell
        {"name": "hpsi_si64_mixed", "op": "hpsi", **cube64, "nb": 160, "prec": "mixed", "prepared": True},
        {"name": "hpsi_si64_fp64", "op": "hpsi", **cube64, "nb": 160, "prec": "fp64"},
        # one k-point of the 255-atom cell with a vacancy, bench.py's headline
        {"name": "hpsi_si255_mixed", "op": "hpsi", **_cell("cubic", 4, 4, 2, 30.0, MP4[0], g1=96, g2=96, g3=48), "vacancy": 1,
         "nb": 288, "prec": "mixed", "prepared": True},
        # the 216-atom cell with real wavefunctions, projectors split on each call
        {"name": "gamma_si216_mixed", "op": "gamma", **_cell("cubic", 3, 3, 3, 20.0), "nb": 480, "prec": "mixed"},
        # many small uneven cells in one replay (screening runs)
        {"name": "batch_64_cells_mixed", "op": "batch", "ncell": 64, "cells_seed": 7, "prec": "mixed"},
        # the Davidson's overlaps and basis rotation on the 64-atom sphere, ragged mid-solve sizes
        {"name": "overlap_480x157_fp64", "op": "zgemm", "product": "cn", "arith": 0, "m": 480, "n": 157, "k": 18232},
        {"name": "rotate_480to157_ds", "op": "zgemm", "product": "tn", "arith": 1, "m": 157, "n": 18232, "k": 480},
        # one time step of a 32-atom cell with an odd band count
        {"name": "etrs_si32_mixed", "op": "etrs", **_cell("cubic", 2, 2, 1, 25.0, MP4[2]), "nb": 81, "prec": "mixed", "dt": 0.05,
         "order": 4, "prepared": True},
        # one (k, k+q) block of GW matrix elements of the 64-atom cell
        {"name": "gw_si64_mixed", "op": "gw", **cube64, "nl": 32, "nr": 64, "eps_frac": 0.25, "prec": "mixed"},
        # the first two self-consistency steps of the 8-atom cell: Davidson solves, densities, potentials
        {"name": "scf_si8_fp64", "op": "scf", **_cell("cubic", 1, 1, 1, 15.0), "nk": 1, "nb": 8, "nelec": 2, "steps": 2, "prec": "fp64"},
        # one training step's loss and gradient of the learned preconditioner
        {"name": "mlp_grad_300k", "op": "mlp", "bands": 300, "npw": 1001},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_cell(rng, most):
    """A supercell of at most `most` atoms with a cutoff of the workloads' range, at a k-point or Gamma."""
    while True:
        kind = rng.choice(("fcc", "cubic"))
        r = sorted((rng.randint(1, 4) for _ in range(3)), reverse=True)
        c = _cell(kind, *r, round(rng.uniform(12, 30), 2), rng.choice(MP4 + ((0.0, 0.0, 0.0),)))
        if _natoms(c) <= most and _nr(c) <= 450_000:
            return c


def draw(rng):
    op = rng.choice(("hpsi", "hpsi", "hpsi", "hpsi", "gamma", "batch", "zgemm", "zgemm", "etrs", "gw", "scf", "mlp"))
    prec = rng.choice(("mixed", "mixed", "fp64"))
    if op in ("hpsi", "gamma", "etrs"):
        c = _draw_cell(rng, 256 if prec == "mixed" and op != "etrs" else 64)
        most = max(4, min(400, 3 * _natoms(c)))
        c.update(op=op, prec=prec, nb=_log(rng, 1 if op != "etrs" else 4, most))
        if op == "gamma":
            c.update(k1=0.0, k2=0.0, k3=0.0)
        if prec == "mixed":
            c["prepared"] = rng.random() < 0.6
        if op == "etrs":
            c.update(dt=round(rng.uniform(0.01, 0.1), 3), order=rng.randint(2, 5))
        return c
    if op == "batch":
        return {"op": op, "ncell": _log(rng, 8, 64), "cells_seed": rng.randint(10, 10 ** 6), "prec": prec}
    if op == "zgemm":
        big, small = _log(rng, 16, 640), _log(rng, 8, 160)
        npw = _log(rng, 400, 40000)
        if rng.random() < 0.5:
            return {"op": op, "product": "cn", "arith": rng.choice((0, 1, 2)), "m": big, "n": small, "k": npw}
        return {"op": op, "product": "tn", "arith": rng.choice((0, 1, 2)), "m": small, "n": npw, "k": big}
    if op == "gw":
        c = _draw_cell(rng, 64)
        c.update(op=op, prec=prec, nl=_log(rng, 1, 24), nr=_log(rng, 4, 48), eps_frac=round(rng.uniform(0.15, 0.5), 3))
        return c
    if op == "scf":
        return {"op": op, **_cell(*rng.choice((("fcc", 1, 1, 1), ("fcc", 2, 1, 1), ("cubic", 1, 1, 1))),
                                  round(rng.uniform(10, 15), 2)),
                "nk": 1, "nb": rng.randint(4, 9), "nelec": 2, "steps": 2, "prec": prec}
    return {"op": op, "bands": _log(rng, 8, 300), "npw": _log(rng, 150, 1001)}


def prepare(case, seed):
    return OPS[case["op"]][0](case, seed)


def run(state):
    return OPS[state["case"]["op"]][1](state)


def exact(case, seed):
    return OPS[case["op"]][2](prepare(case, seed))


def work(case):
    return OPS[case["op"]][3](case)
