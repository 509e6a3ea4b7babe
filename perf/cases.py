"""Workloads of the Fock-like exchange library, as a program calls it.

A case is a dict of plain values:

  op      apply | energy | vjp (autograd, forward and backward) | step | ortho | batched
  dtype   c64 (fused FP32 form) or c128 (FP64 form)
  grid    "n1xn2xn3"        k   "n1xn2xn3" Monkhorst-Pack mesh
  occ     occupied bands    tgt  target bands (apply, vjp)
  q       "m1xm2xm3" mesh of the down-sampled Fock sum, or "" for every k-point (apply)
  smear   occupations drawn from (0, 1] with some empty bands, instead of all 1
  cells   batched: number of uneven cells, drawn from `pick`

Orbitals are seeded random plane waves below a 6 Ha cutoff on the 10.26 bohr silicon-like
cubic cell, orthonormalised per k-point: the structure a ground state has.  `work` counts a
pair convolution as one forward and one inverse 3-D FFT of 5 N log2 N flops each.
"""
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_1507_05156_gb300 import hse, tdks

A_CELL = 10.26          # bohr
OMEGA, ALPHA, SPIN = 0.106, 0.25, 2.0
ECUT = 6.0              # Ha
A_VEC = (0.01, -0.004, 0.007)  # vector potential of the step cases (bohr^-1)
DT = 0.04               # time step of the paper's runs (a.u.)


def _case(name, op, grid, k, occ, tgt=0, dtype="c64", q="", smear=False, cells=0, pick=0):
    c = {"op": op, "dtype": dtype, "grid": grid, "k": k, "occ": occ, "tgt": tgt or occ, "q": q, "smear": smear,
         "cells": cells, "pick": pick}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call in use: a coarse toy cell in a test or a notebook, all latency
        _case("apply_8_k2_b4", "apply", "8x8x8", "2x2x2", 4),
        # the FP64 form on the small validation workload
        _case("apply_12_k2_b4_fp64", "apply", "12x12x12", "2x2x2", 4, dtype="c128"),
        # the paper's silicon run: 16^3 grid, 12^3 k-points, the Fock sum over a 4^3 mesh, 16 bands
        _case("apply_16_k12_q4_b16", "apply", "16x16x16", "12x12x12", 16, q="4x4x4"),
        # a ragged cell: uneven mesh, odd band counts, partly filled and empty bands
        _case("apply_18_k321_b7+9", "apply", "18x18x18", "3x2x1", 7, tgt=9, smear=True),
        # one Hamiltonian application of an ordinary ground-state or time-propagation run
        _case("apply_20_k4_b16", "apply", "20x20x20", "4x4x4", 16),
        # the finest grid, occupied and empty target bands (the benchmark's cell on a 4^3 mesh)
        _case("apply_24_k4_b16+16", "apply", "24x24x24", "4x4x4", 16, tgt=32),
        # the exchange part of a total energy, in FP64
        _case("energy_16_k2_b8_fp64", "energy", "16x16x16", "2x2x2", 8, dtype="c128"),
        # V_x u and its three gradients: the differentiation workload, and a fine-grid cell
        _case("vjp_16_k3_b8", "vjp", "16x16x16", "3x3x3", 8),
        _case("vjp_24_k2_b8", "vjp", "24x24x24", "2x2x2", 8),
        # one time step with its observables: current, Hartree potential, Taylor step, overlaps
        _case("step_16_k3_b8", "step", "16x16x16", "3x3x3", 8),
        # orthonormalising a start set
        _case("ortho_20_k4_b16", "ortho", "20x20x20", "4x4x4", 16),
        # a batch of uneven small cells in one call
        _case("batched_10", "batched", "", "", 0, cells=10, pick=3),
    ]


SIDES = (4, 6, 8, 10, 12, 16, 18, 20, 24)
AXES_FP64 = (4, 5, 6, 8, 9, 10, 12, 15, 16, 18, 20)


def draw(rng: random.Random):
    while True:
        op = rng.choice(["apply"] * 5 + ["energy", "energy", "vjp", "vjp", "step", "ortho", "batched"])
        if op == "batched":
            return _case("", op, "", "", 0, cells=rng.randint(2, 10), pick=rng.randrange(1 << 20))
        dtype = "c128" if op == "energy" or rng.random() < 0.25 else "c64"
        if dtype == "c64":
            n = rng.choice(SIDES)
            grid = (n, n, n)
        else:
            grid = tuple(rng.choice(AXES_FP64) for _ in range(3))
            if rng.random() < 0.5:
                grid = (grid[0],) * 3
        q = ""
        if op == "apply" and rng.random() < 0.2:
            m = tuple(rng.randint(1, 2) for _ in range(3))
            k = tuple(3 * v for v in m)
            q = "x".join(map(str, m))
        else:
            k = tuple(rng.randint(1, 4) for _ in range(3))
        occ = round(2 ** rng.uniform(0, 4))
        tgt = occ if op in ("energy", "step", "ortho") else max(1, round(2 ** rng.uniform(0, 5)))
        if rng.random() < 0.5:
            tgt = occ
        c = _case("", op, "x".join(map(str, grid)), "x".join(map(str, k)), occ, tgt, dtype, q, rng.random() < 0.25)
        if work(c)["flops"] <= (1.5e10 if dtype == "c128" else 1.5e12):
            return c


# ---------------------------------------------------------------- inputs

def _ints(text):
    return tuple(int(v) for v in text.split("x"))


def _mesh(n):
    """Cartesian Monkhorst-Pack points of the cubic cell, first axis slowest."""
    b = 2.0 * math.pi / A_CELL
    ax = [[(2.0 * r - m - 1.0) / (2.0 * m) * b for r in range(1, m + 1)] for m in n]
    return np.array([(x, y, z) for x in ax[0] for y in ax[1] for z in ax[2]])


def _submesh(n, m):
    """Indices in _mesh(n) of the points of _mesh(m); each n_d is an odd multiple of m_d."""
    ax = [[(nd // md) * r + (nd // md - 1) // 2 for r in range(md)] for nd, md in zip(n, m)]
    return [(x * n[1] + y) * n[2] + z for x in ax[0] for y in ax[1] for z in ax[2]]


def _gvec(grid):
    """G vectors [N][3] (float64, on the GPU), FFT order, the Nyquist index negative."""
    b = 2.0 * math.pi / A_CELL
    ax = [torch.tensor([(i if i <= (n - 1) // 2 else i - n) * b for i in range(n)], dtype=torch.float64) for n in grid]
    return torch.stack(torch.meshgrid(*ax, indexing="ij"), -1).reshape(-1, 3).cuda()


def _orbitals(gen, grid, kpts, nb, dtype, orthonormal=True):
    N, nk = math.prod(grid), len(kpts)
    dV = A_CELL ** 3 / N
    G = _gvec(grid)
    out = torch.empty((nk, nb) + grid, dtype=dtype, device="cuda")
    step = max(1, (1 << 24) // (nb * N))
    for k0 in range(0, nk, step):
        kk = torch.as_tensor(kpts[k0:k0 + step], device="cuda")
        inside = ((G[None] + kk[:, None]) ** 2).sum(-1) < 2.0 * ECUT
        c = torch.randn((len(kk), nb, N), dtype=torch.complex128, device="cuda", generator=gen) * inside[:, None]
        if orthonormal:
            L = torch.linalg.cholesky(c @ c.mH)
            c = torch.linalg.solve_triangular(L, c, upper=False)
        else:
            c = c / torch.linalg.vector_norm(c, dim=-1, keepdim=True)
        u = torch.fft.ifftn(c.reshape((len(kk), nb) + grid), dim=(2, 3, 4)) * (N / math.sqrt(N * dV))
        out[k0:k0 + step] = u
    return out


def _occupations(gen, nk, n_occ, smear):
    if not smear:
        return torch.ones((nk, n_occ), dtype=torch.float64, device="cuda")
    f = torch.rand((nk, n_occ), dtype=torch.float64, device="cuda", generator=gen) * 1.1
    f = torch.where(f > 1.0, torch.zeros_like(f), 1.0 - f)
    return f


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _inputs(case, seed):
    """The tensors of a single-cell case."""
    gen = _gen(seed)
    grid, mesh = _ints(case["grid"]), _ints(case["k"])
    s = SimpleNamespace(grid=grid, kpts=_mesh(mesh), dtype=torch.complex64 if case["dtype"] == "c64" else torch.complex128,
                        kocc=_submesh(mesh, _ints(case["q"])) if case["q"] else None, n_occ=case["occ"], n_tgt=case["tgt"])
    nk = len(s.kpts)
    if case["op"] == "ortho":
        s.u = _orbitals(gen, grid, s.kpts, case["occ"], s.dtype, orthonormal=False)
        return s
    u = _orbitals(gen, grid, s.kpts, max(s.n_occ, s.n_tgt), s.dtype)
    s.u_occ = u[:, :s.n_occ].contiguous()
    s.u_tgt = s.u_occ if s.n_tgt == s.n_occ else u[:, :s.n_tgt].contiguous()
    s.occ = _occupations(gen, nk, s.n_occ, case["smear"])
    if case["op"] == "vjp":  # the cotangent of an energy-like loss and a random one
        s.ybar = torch.randn(s.u_tgt.shape, dtype=s.dtype, device="cuda", generator=gen) * s.u_tgt.abs().mean() - s.u_tgt
    return s


def _omega(case):
    """omega as the program holds it: a parameter of the orbitals' precision where it is differentiated."""
    return torch.tensor(OMEGA, dtype=torch.float32 if case["op"] == "vjp" and case["dtype"] == "c64" else torch.float64)


def _cells(case, seed):
    """The uneven cells of a batched case (grids, meshes and bands as the batched workload draws them)."""
    r = random.Random(case["pick"])
    gen = _gen(seed)
    cells = []
    for _ in range(case["cells"]):
        n, m, nb = r.choice((12, 16, 18, 20, 24)), r.choice((2, 3)), r.randint(4, 16)
        s = SimpleNamespace(grid=(n, n, n), kpts=_mesh((m, m, m)), n_occ=nb, n_tgt=nb, lattice=np.eye(3) * A_CELL,
                            omega=OMEGA, alpha=ALPHA, kocc=None)
        s.u_occ = s.u_tgt = _orbitals(gen, s.grid, s.kpts, nb, torch.complex64)
        s.occ = torch.ones((m ** 3, nb), dtype=torch.float64, device="cuda")
        cells.append(s)
    return cells


def prepare(case, seed):
    if case["op"] == "batched":
        cells = _cells(case, seed)
        return {"op": "batched", "plan": hse.BatchedPlan(cells), "u_occ": [c.u_occ for c in cells],
                "occ": [c.occ for c in cells], "u_tgt": [c.u_tgt for c in cells]}
    s = _inputs(case, seed)
    if case["op"] == "vjp":
        geom = tdks.Geometry(s.grid, np.eye(3) * A_CELL, s.kpts, ALPHA, SPIN)
        omega = _omega(case).requires_grad_()
        leaves = (s.u_occ.requires_grad_(), s.u_tgt.detach().requires_grad_(), omega)
        return {"op": "vjp", "geom": geom, "plan": geom.plan(s.n_occ, s.n_tgt, omega, s.dtype), "leaves": leaves,
                "occ": s.occ, "ybar": s.ybar}
    plan = hse.Plan(s.grid, np.eye(3) * A_CELL, s.kpts, s.n_occ, s.n_tgt, OMEGA, ALPHA, SPIN, dtype=s.dtype, kocc=s.kocc)
    return dict(vars(s), op=case["op"], plan=plan)


def run(state):
    op, plan = state["op"], state["plan"]
    if op == "apply":
        return hse.hse_fock_apply(plan, state["u_occ"], state["occ"], state["u_tgt"])
    if op == "energy":
        return hse.hse_exchange_energy(plan, state["u_occ"], state["occ"])
    if op == "vjp":
        u_occ, u_tgt, omega = state["leaves"]
        vx = tdks.fock_apply(u_occ, state["occ"], u_tgt, omega, state["geom"])
        loss = (vx * state["ybar"].conj()).real.sum()  # its cotangent with respect to vx is ybar
        return vx.detach(), torch.autograd.grad(loss, state["leaves"])
    if op == "step":
        psi, occ = state["u_occ"], state["occ"]
        J = hse.hse_current(plan, psi, occ, A_VEC)
        vh = hse.hse_hartree_potential(plan, psi, occ)
        S = hse.hse_overlap(plan, psi)
        return {"psi": hse.hse_taylor_step(plan, psi, occ, A_VEC, DT, vloc=vh), "J": J, "vh": vh, "S": S}
    if op == "ortho":
        return hse.hse_orthonormalize(plan, state["u"].clone())
    return hse.hse_fock_apply_batched(plan, state["u_occ"], state["occ"], state["u_tgt"])


def _pair_flops(N):
    return 10.0 * N * math.log2(N) + 16.0 * N


def work(case):
    if case["op"] == "batched":
        r = random.Random(case["pick"])
        b = f = 0.0
        for _ in range(case["cells"]):
            n, m, nb = r.choice((12, 16, 18, 20, 24)), r.choice((2, 3)), r.randint(4, 16)
            f += (m ** 3 * nb) ** 2 * _pair_flops(n ** 3)
            b += m ** 3 * nb * n ** 3 * 8 * 2
        return {"bytes": b, "flops": f}
    N, nk = math.prod(_ints(case["grid"])), math.prod(_ints(case["k"]))
    nq = math.prod(_ints(case["q"])) if case["q"] else nk
    eb = 8 if case["dtype"] == "c64" else 16
    occ, tgt, op = case["occ"], case["tgt"], case["op"]
    orb = nk * N * eb  # one band
    pairs = nk * tgt * nq * occ
    same = 0 if tgt == occ else tgt
    if op == "apply":
        return {"bytes": orb * (tgt + (same and tgt)) + nq * occ * N * eb, "flops": pairs * _pair_flops(N)}
    if op == "energy":  # sum_G v |rho(G)|^2 over the unordered pairs: one forward transform each
        return {"bytes": orb * occ, "flops": 0.5 * pairs * (5.0 * N * math.log2(N) + 10.0 * N)}
    if op == "vjp":     # two convolutions a pair (of u_i and of ybar_i), the u_occ gradient's products besides
        return {"bytes": orb * (2 * occ + 3 * tgt + same), "flops": 2.0 * pairs * (_pair_flops(N) + 8.0 * N)}
    if op == "step":    # four applications, the transforms of T and J
        return {"bytes": 2.0 * orb * occ, "flops": 4.0 * pairs * _pair_flops(N) + 45.0 * nk * occ * N * math.log2(N)}
    return {"bytes": 2.0 * orb * occ, "flops": 8.0 * nk * occ * (occ + 1) * N}  # ortho


# ---------------------------------------------------------------- the same in 64 bits, plain torch

def _v(grid, q, omega=OMEGA):
    """v(|G+q|) and its derivative with respect to omega on the grid."""
    g2 = ((_gvec(grid) + torch.as_tensor(q, device="cuda")) ** 2).sum(-1)
    x = g2 / (4.0 * omega ** 2)
    lim = math.pi / omega ** 2
    v = torch.where(x == 0, torch.full_like(x, lim), lim * -torch.expm1(-x) / torch.where(x == 0, torch.ones_like(x), x))
    dv = -(2.0 * math.pi / omega ** 3) * torch.exp(-x)
    return v.reshape(grid), dv.reshape(grid)


_DIMS = (-3, -2, -1)


def _rows(s):
    return list(range(len(s.kpts))) if s.kocc is None else list(s.kocc)


def _conv(rho, v):
    return torch.fft.ifftn(torch.fft.fftn(rho, dim=_DIMS) * v, dim=_DIMS)


def _fock(s, u_occ, u_tgt):
    """V_x u_tgt (complex128): -alpha/N_q sum f u_j K_q(conj(u_j) u_i)."""
    rows = _rows(s)
    out = torch.zeros_like(u_tgt)
    chunk = max(1, (1 << 25) // (u_occ.shape[1] * math.prod(s.grid)))
    for k in range(len(s.kpts)):
        for kp in rows:
            v, _ = _v(s.grid, s.kpts[k] - s.kpts[kp])
            uj, f = u_occ[kp][None], s.occ[kp].reshape(1, -1, 1, 1, 1)
            for i in range(0, u_tgt.shape[1], chunk):
                phi = _conv(uj.conj() * u_tgt[k, i:i + chunk, None], v)
                out[k, i:i + chunk] -= ALPHA / len(rows) * (f * uj * phi).sum(1)
    return out


def _vjp(s, u_occ, u_tgt, y, omega):
    vx, g_occ, g_tgt = torch.zeros_like(u_tgt), torch.zeros_like(u_occ), torch.zeros_like(u_tgt)
    g_om = torch.zeros((), dtype=torch.float64, device="cuda")
    chunk = max(1, (1 << 24) // (u_occ.shape[1] * math.prod(s.grid)))
    for k in range(len(s.kpts)):
        for kp in range(len(s.kpts)):
            v, dv = _v(s.grid, s.kpts[k] - s.kpts[kp], omega)
            uj = u_occ[kp][None]
            c = ALPHA / len(s.kpts) * s.occ[kp].reshape(1, -1, 1, 1, 1)
            for i in range(0, u_tgt.shape[1], chunk):
                ui, yi = u_tgt[k, i:i + chunk, None], y[k, i:i + chunk, None]
                a = torch.fft.fftn(uj.conj() * ui, dim=_DIMS)
                b = torch.fft.fftn(uj.conj() * yi, dim=_DIMS)
                phi, psi = torch.fft.ifftn(a * v, dim=_DIMS), torch.fft.ifftn(b * v, dim=_DIMS)
                vx[k, i:i + chunk] -= (c * uj * phi).sum(1)
                g_tgt[k, i:i + chunk] -= (c * uj * psi).sum(1)
                g_occ[kp] -= (c * (phi.conj() * yi + ui * psi.conj())).sum(0)
                g_om -= (c * dv * (a * b.conj()).real).sum() / math.prod(s.grid)
    return vx, (g_occ, g_tgt, g_om)


def _step(s, psi):
    grid, N, nk = s.grid, math.prod(s.grid), len(s.kpts)
    G = _gvec(grid)
    w = (SPIN / nk * s.occ).reshape(nk, -1, 1, 1, 1)
    kA = torch.as_tensor(s.kpts + np.array(A_VEC), device="cuda")
    gka = G[None] + kA[:, None]                                     # [nk][N][3]
    c2 = (torch.fft.fftn(psi, dim=_DIMS) / N).abs().square().reshape(nk, -1, N)
    J = -torch.einsum("kb,kbg,kgc->c", w.reshape(nk, -1), c2, gka)
    rho = (w * psi.abs().square()).sum((0, 1))
    g2 = (G ** 2).sum(-1).reshape(grid)
    vh = torch.fft.ifftn(torch.fft.fftn(rho.to(torch.complex128)) *
                         torch.where(g2 > 0, 4.0 * math.pi / torch.where(g2 > 0, g2, torch.ones_like(g2)), 0.0)).real
    kin = 0.5 * (gka ** 2).sum(-1).reshape((nk, 1) + grid)
    out, term = psi.clone(), psi
    for n in range(1, 5):
        h = _conv(term, kin) + vh * term + _fock(s, psi, term)
        term = (-1j * DT / n) * h
        out = out + term
    flat = psi.reshape(nk, -1, N)
    S = (flat.conj() @ flat.transpose(1, 2)) * (A_CELL ** 3 / N)
    return {"psi": out, "J": J, "vh": vh, "S": S}


def exact(case, seed):
    op = case["op"]
    if op == "batched":
        if work(case)["flops"] > 3e12:
            return None
        return [_fock(c, c.u_occ.to(torch.complex128), c.u_tgt.to(torch.complex128)) for c in _cells(case, seed)]
    nk = math.prod(_ints(case["k"]))
    nq = math.prod(_ints(case["q"])) if case["q"] else nk
    if work(case)["flops"] > 6e12 or nk * nq > 8000:
        return None  # the largest mesh: over a minute
    s = _inputs(case, seed)
    wide = lambda t: t.to(torch.complex128)  # noqa: E731
    if op == "ortho":
        N = math.prod(s.grid)
        flat = wide(s.u).reshape(nk, -1, N)
        L = torch.linalg.cholesky((flat @ flat.mH) * (A_CELL ** 3 / N))
        return torch.linalg.solve_triangular(L, flat, upper=False).reshape(s.u.shape)
    u_occ = wide(s.u_occ)
    if op == "apply":
        return _fock(s, u_occ, wide(s.u_tgt))
    if op == "energy":
        vx = _fock(s, u_occ, u_occ)
        dV = A_CELL ** 3 / math.prod(s.grid)
        return 0.5 * SPIN / nk * dV * (s.occ.reshape(nk, -1, 1, 1, 1) * (u_occ.conj() * vx).real).sum()
    if op == "vjp":
        return _vjp(s, u_occ, wide(s.u_tgt), wide(s.ybar), float(_omega(case)))
    return _step(s, u_occ)
