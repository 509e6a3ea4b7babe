"""The two-exchange 16^3 kernel (four owners a CTA, 64 points a thread) at its edges, against the
FP64 oracle: tiles with one to four owners, one partner, partners skipped at both ends of a k'
and over a whole k' (the kernel row and the stage buffers advance past them), more partners than
the occupation cache holds, and a split k' range (few tiles, many partners).

Tolerance 1e-5 (relative L2), the complex64 bound of the parity tests: each 3-D transform of 4096
points has a relative rms error of about eps log2 N = 7e-7, the sums add a few eps.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1507_05156_gb300 import hse, inputs

pytestmark = pytest.mark.gpu

# nk, n_occ, n_tgt, empties: (k', band) ranges set to f = 0
CASES = [(1, 1, 1, ()), (1, 2, 3, ()), (2, 3, 4, ((0, 0), (1, 2))), (3, 2, 5, ((1, 0), (1, 1))),
         (2, 17, 2, ((0, 16), (1, 0))), (7, 4, 9, ((0, 0), (0, 1), (0, 2), (0, 3), (6, 3))), (4, 260, 1, ((2, 5),))]


@pytest.mark.parametrize("nk,n_occ,n_tgt,empty", CASES)
def test_wide_apply(nk, n_occ, n_tgt, empty, monkeypatch):
    monkeypatch.setenv("HSE_BLOCKS_PER_SM", "6")  # small plans choose the staged-partner kernel by themselves
    grid = (16, 16, 16)
    lattice = inputs.cubic_lattice(inputs.A_SI)
    rng = np.random.default_rng(1600 + 10 * nk + n_tgt)
    kpts = (rng.random((nk, 3)) - 0.5) @ (2 * np.pi * np.linalg.inv(lattice).T)
    c64 = lambda s, shape: (inputs.random_orbitals(s, shape) * 0.06).astype(np.complex64)  # noqa: E731
    u_occ, u_tgt = c64(nk + 1, (nk, n_occ) + grid), c64(nk + 2, (nk, n_tgt) + grid)
    occ = 0.5 + 0.5 * rng.random((nk, n_occ))
    for k, j in empty:
        occ[k, j] = 0.0
    plan = hse.Plan(grid, lattice, kpts, n_occ, n_tgt, inputs.OMEGA, inputs.ALPHA, dtype=torch.complex64)
    out = hse.hse_fock_apply(plan, torch.from_numpy(u_occ).cuda(), torch.from_numpy(occ).cuda(),
                             torch.from_numpy(u_tgt).cuda())
    hse.hse_status(plan)
    ref = oracle.fock_apply(u_occ.astype(np.complex128), occ, u_tgt.astype(np.complex128), kpts, lattice, grid,
                            inputs.OMEGA, inputs.ALPHA)
    ybar = c64(nk + 3, u_tgt.shape)
    for omega in (True, False):  # with and without the omega gradient riding on the u_occ pass
        g_occ, _, g_om = hse.hse_fock_apply_vjp(plan, torch.from_numpy(u_occ).cuda(), torch.from_numpy(occ).cuda(),
                                                torch.from_numpy(u_tgt).cuda(), torch.from_numpy(ybar).cuda(), need_omega=omega)
        hse.hse_status(plan)
        w = [x.astype(np.complex128) for x in (u_occ, u_tgt, ybar)]
        r_occ, _, r_om = oracle.fock_apply_vjp(w[0], occ, w[1], w[2], kpts, lattice, grid, inputs.OMEGA, inputs.ALPHA)
        assert np.linalg.norm(g_occ.cpu().numpy() - r_occ) <= 1e-5 * np.linalg.norm(r_occ)
        if omega:  # a sum of terms of both signs: against its Cauchy-Schwarz scale
            dvx = oracle.fock_apply(w[0], occ, w[1], kpts, lattice, grid, inputs.OMEGA, inputs.ALPHA, kernel="domega")
            assert abs(g_om.item() - r_om) <= 1e-5 * np.linalg.norm(w[2]) * np.linalg.norm(dvx)
    got = out.cpu().numpy().astype(np.complex128)
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)
    for k in range(nk):
        for i in range(n_tgt):
            assert np.linalg.norm(got[k, i] - ref[k, i]) <= 3e-5 * np.linalg.norm(ref[k, i])
