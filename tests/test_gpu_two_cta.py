"""The two-CTA pencil-load kernel of the 18^3 and 20^3 apply (one pencil per thread, the last warp
half empty) against the FP64 oracle: one and several owners, skipped partners, split ranges, more
k-points than a fold group, and the caller's layout instead of the pencil-blocked copies.
Tolerance 1e-5, the complex64 bound of the parity tests.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1507_05156_gb300 import hse, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nk,n_occ,n_tgt,blocks", [(18, 1, 1, 1, 1), (18, 3, 3, 2, 1), (18, 2, 17, 1, 0), (20, 1, 1, 2, 1),
                                                     (20, 9, 2, 1, 1), (20, 2, 17, 3, 1), (20, 2, 2, 2, 0)])
def test_two_cta_apply(n, nk, n_occ, n_tgt, blocks, monkeypatch):
    monkeypatch.setenv("HSE_BLOCKS_PER_SM", "7")
    monkeypatch.setenv("HSE_PENCIL_BLOCKS", str(blocks))
    grid = (n, n, n)
    lattice = inputs.cubic_lattice(inputs.A_SI)
    rng = np.random.default_rng(n + 10 * nk + n_occ)
    kpts = (rng.random((nk, 3)) - 0.5) @ (2 * np.pi * np.linalg.inv(lattice).T)
    c64 = lambda s, shape: (inputs.random_orbitals(s, shape) * 0.06).astype(np.complex64)  # noqa: E731
    u_occ, u_tgt = c64(nk + 1, (nk, n_occ) + grid), c64(nk + 2, (nk, n_tgt) + grid)
    occ = 0.5 + 0.5 * rng.random((nk, n_occ))
    if n_occ > 1:
        occ[0, 0] = occ[-1, -1] = 0.0
    plan = hse.Plan(grid, lattice, kpts, n_occ, n_tgt, inputs.OMEGA, inputs.ALPHA, dtype=torch.complex64)
    out = hse.hse_fock_apply(plan, torch.from_numpy(u_occ).cuda(), torch.from_numpy(occ).cuda(),
                             torch.from_numpy(u_tgt).cuda())
    hse.hse_status(plan)
    ref = oracle.fock_apply(u_occ.astype(np.complex128), occ, u_tgt.astype(np.complex128), kpts, lattice, grid,
                            inputs.OMEGA, inputs.ALPHA)
    assert np.linalg.norm(out.cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref)
