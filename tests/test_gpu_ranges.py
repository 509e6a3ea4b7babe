"""Partner ranges of every length, and tiles of every size, forced through the plan's test hooks
(HSE_RANGES: how many ranges; HSE_F64_TILE: orbitals a CTA of the fused FP64 passes), so that what the
estimates seldom choose is checked too: items with more partners than the occupation cache holds,
empty bands past its end, ranges that start inside a k-point, many fold groups in an item, FP64 tiles
that straddle k-points and end partly filled.  References and tolerances are those of the parity tests
(1e-5 complex64, 1e-10 complex128, relative L2) and of the compensated sums.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1507_05156_gb300 import hse, inputs
from test_gpu_compensated import TOL, _copies, _dev, _max_rel

pytestmark = pytest.mark.gpu

LATTICE = inputs.cubic_lattice(inputs.A_SI)


def _problem(n, nk, n_occ, n_tgt):
    grid = (n,) * 3
    rng = np.random.default_rng(n + 31 * nk + n_occ)
    kpts = (rng.random((nk, 3)) - 0.5) @ (2 * np.pi * np.linalg.inv(LATTICE).T)
    c64 = lambda s, nb: (inputs.random_orbitals(s, (nk, nb) + grid) * 0.06).astype(np.complex64)  # noqa: E731
    return grid, kpts, c64(nk + 1, n_occ), c64(nk + 2, n_tgt), c64(nk + 3, n_tgt), 0.5 + 0.5 * rng.random((nk, n_occ))


def _plan(p, monkeypatch, variant, ranges):
    monkeypatch.setenv("HSE_BLOCKS_PER_SM", str(variant))
    monkeypatch.setenv("HSE_RANGES", str(ranges))
    return hse.Plan(p[0], LATTICE, p[1], p[2].shape[1], p[3].shape[1], inputs.OMEGA, inputs.ALPHA)


def _rel(a, b):
    return np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b)


# staged kernel (0, -1, -2) and two-exchange kernel (6); 2 ranges of 3 x 800: the second starts inside k' = 1
@pytest.mark.parametrize("n,variant", [(4, 0), (8, -1), (8, -2), (16, 6), (16, -1)])
@pytest.mark.parametrize("nk,n_occ,ranges", [(1, 1100, 1), (3, 800, 2)])
def test_more_partners_than_the_occupation_cache(n, variant, nk, n_occ, ranges, monkeypatch):
    p = _problem(n, nk, n_occ, 1)
    occ = p[5]
    occ[:, ::7] = 0.0
    occ[-1, -3:] = 0.0
    occ[0, 0] = 0.0
    if nk > 1:
        occ[1, 390:410] = 0.0  # around the start of the second range
        occ[2, :300] = 0.0
    plan = _plan(p, monkeypatch, variant, ranges)
    out = hse.hse_fock_apply(plan, torch.from_numpy(p[2]).cuda(), torch.from_numpy(occ).cuda(), torch.from_numpy(p[3]).cuda())
    hse.hse_status(plan)
    ref = oracle.fock_apply(p[2].astype(np.complex128), occ, p[3].astype(np.complex128), p[1], LATTICE, p[0], inputs.OMEGA, inputs.ALPHA)
    assert _rel(out, ref) <= 1e-5


@pytest.mark.parametrize("n,variant", [(8, -1), (8, 7), (12, 7), (16, 6), (18, 7), (18, -2), (20, 7), (24, 0)])
@pytest.mark.parametrize("nk,n_occ,n_tgt,ranges", [(5, 16, 2, 1), (5, 2, 16, 1), (5, 3, 16, 2), (9, 9, 1, 2)])
def test_fold_groups(n, variant, nk, n_occ, n_tgt, ranges, monkeypatch):
    """Up to five groups an item in the apply (16 occupied bands) and in the u_occ pass (16 targets)."""
    p = _problem(n, nk, n_occ, n_tgt)
    grid, kpts, u_occ, u_tgt, ybar, occ = p
    occ[nk // 2] = 0.0  # a whole k'
    plan = _plan(p, monkeypatch, variant, ranges)
    d = [torch.from_numpy(a).cuda() for a in (u_occ, occ, u_tgt, ybar)]
    out = hse.hse_fock_apply(plan, *d[:3])
    g_occ, _, g_om = hse.hse_fock_apply_vjp(plan, *d, need_tgt=False)
    g_occ2, _, _ = hse.hse_fock_apply_vjp(plan, *d, need_tgt=False, need_omega=False)
    g_om2 = hse.hse_fock_apply_vjp(plan, *d, need_occ=False, need_tgt=False)[2]
    e = hse.hse_exchange_energy(plan, d[0], d[1])
    hse.hse_status(plan)
    w = [a.astype(np.complex128) for a in (u_occ, u_tgt, ybar)]
    args = (kpts, LATTICE, grid, inputs.OMEGA, inputs.ALPHA)
    assert _rel(out, oracle.fock_apply(w[0], occ, w[1], *args)) <= 1e-5
    r_occ, _, r_om = oracle.fock_apply_vjp(w[0], occ, w[1], w[2], *args)
    assert _rel(g_occ, r_occ) <= 1e-5 and _rel(g_occ2, r_occ) <= 1e-5
    scale = np.linalg.norm(w[2]) * np.linalg.norm(oracle.fock_apply(w[0], occ, w[1], *args, kernel="domega"))
    assert abs(g_om.item() - r_om) <= 1e-5 * scale and abs(g_om2.item() - r_om) <= 1e-5 * scale
    e_ref = oracle.exchange_energy(w[0], occ, *args, 2.0)
    assert abs(e.item() - e_ref) <= 1e-5 * abs(e_ref)


@pytest.mark.parametrize("n,variant", [(16, 6), (18, 7), (20, 7)])
def test_sum_over_copies(n, variant, monkeypatch):
    """512 equal k-points in one range (see test_gpu_compensated.py): the running sums of the
    two-exchange and the two-CTA kernel do not drift."""
    monkeypatch.setenv("HSE_BLOCKS_PER_SM", str(variant))
    monkeypatch.setenv("HSE_RANGES", "1")
    grid, lattice, k0, u_occ1, u_tgt1, ybar1, occ1, kpts, u_occ, u_tgt, ybar, occ = _copies(n, 2, 1, 40 + n)
    d = torch.complex64
    plan = hse.Plan(grid, lattice, kpts, 2, 1, inputs.OMEGA, inputs.ALPHA, dtype=d)
    a = _dev(u_occ, d), _dev(occ, torch.float64), _dev(u_tgt, d)
    out = hse.hse_fock_apply(plan, *a)
    g_occ = hse.hse_fock_apply_vjp(plan, *a, _dev(ybar, d), need_tgt=False, need_omega=False)[0]
    hse.hse_status(plan)
    args = (k0, lattice, grid, inputs.OMEGA, inputs.ALPHA)
    assert _max_rel(out.cpu().numpy(), oracle.fock_apply(u_occ1, occ1, u_tgt1, *args)) <= TOL
    assert _max_rel(g_occ.cpu().numpy(), oracle.fock_apply_vjp(u_occ1, occ1, u_tgt1, ybar1, *args)[0]) <= TOL


# grid, nk, n_occ, n_tgt, kocc: 9, 10, 21 and 16 owners of the energy, tiles across k-points
@pytest.mark.parametrize("grid,nk,n_occ,n_tgt,kocc", [((4, 3, 5), 3, 3, 5, None), ((6, 4, 5), 2, 5, 3, None),
                                                      ((8, 8, 8), 3, 7, 2, (0, 2)), ((5, 6, 4), 4, 4, 1, None),
                                                      ((9, 4, 6), 1, 1, 17, None)])
@pytest.mark.parametrize("tile", [2, 4, 16])
@pytest.mark.parametrize("ranges", [1, 3])
def test_fused_f64_tiles(grid, nk, n_occ, n_tgt, kocc, tile, ranges, monkeypatch):
    monkeypatch.setenv("HSE_FP64_FUSED", "1")
    monkeypatch.setenv("HSE_F64_TILE", str(tile))
    monkeypatch.setenv("HSE_RANGES", str(ranges))
    lattice = np.array([[7.1, 0.3, -0.4], [0.9, 6.2, 0.5], [-0.6, 1.1, 5.3]])
    rng = np.random.default_rng(sum(grid) + 100 * nk + n_tgt)
    kpts = (rng.random((nk, 3)) - 0.5) @ (2 * np.pi * np.linalg.inv(lattice).T)
    u_occ, u_tgt, ybar = (inputs.random_orbitals(s, (nk, nb) + grid) * 0.1 for s, nb in ((1, n_occ), (2, n_tgt), (3, n_tgt)))
    occ = rng.random((nk, n_occ))
    occ[0, -1] = 0.0
    ks = None if kocc is None else list(kocc)
    kw = {} if ks is None else {"kocc": ks}
    plan = hse.Plan(grid, lattice, kpts, n_occ, n_tgt, 0.2, 0.25, dtype=torch.complex128, kocc=ks)
    d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (u_occ, occ, u_tgt, ybar)]
    args = (kpts, lattice, grid, 0.2, 0.25)
    if nk * n_occ > 1:
        e = hse.hse_exchange_energy(plan, d[0], d[1]).item()
        e_ref = oracle.exchange_energy(u_occ, occ, *args, 2.0, **kw)
        assert abs(e - e_ref) <= 1e-10 * abs(e_ref)
        assert _rel(hse.hse_fock_apply(plan, *d[:3]), oracle.fock_apply(u_occ, occ, u_tgt, *args, **kw)) <= 1e-10
        g = hse.hse_fock_apply_vjp(plan, *d)
        r = oracle.fock_apply_vjp(u_occ, occ, u_tgt, ybar, *args, **kw)
        assert _rel(g[0], r[0]) <= 1e-10 and _rel(g[1], r[1]) <= 1e-10 and abs(g[2].item() - r[2]) <= 1e-10 * abs(r[2])
    else:  # the only band is empty
        assert hse.hse_exchange_energy(plan, d[0], d[1]).item() == 0.0
        assert not hse.hse_fock_apply(plan, *d[:3]).abs().any()
    hse.hse_status(plan)
