"""The two-CTA pencil-load kernel of the apply (one pencil per thread, the last warp half empty at 18^3
and 20^3, several owner slots a CTA up to 12^3) against the FP64 oracle: one and several owners, skipped
partners, split ranges, more k-points than a fold group, and the caller's layout instead of the
pencil-blocked copies.  Tolerance 1e-5, the complex64 bound of the parity tests.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1507_05156_gb300 import hse, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nk,n_occ,n_tgt,blocks", [(18, 1, 1, 1, 1), (18, 3, 3, 2, 1), (18, 2, 17, 1, 0), (20, 1, 1, 2, 1),
                                                     (20, 9, 2, 1, 1), (20, 2, 17, 3, 1), (20, 2, 2, 2, 0),
                                                     (8, 2, 3, 9, 1), (8, 3, 1, 1, 0), (10, 2, 2, 5, 1), (10, 3, 3, 4, 0),
                                                     (12, 2, 3, 5, 1), (12, 1, 17, 2, 0)])
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


def test_first_apply_is_captured(monkeypatch):
    """A plan's first apply, captured into a graph, allocates nothing and gives what a call gives."""
    monkeypatch.setenv("HSE_BLOCKS_PER_SM", "7")
    n, nk, nb = 18, 2, 2
    lattice = inputs.cubic_lattice(inputs.A_SI)
    kpts = np.array([[0.0, 0.0, 0.0], [0.1, 0.0, 0.2]])
    u = torch.from_numpy(inputs.random_orbitals(5, (nk, nb, n, n, n)).astype(np.complex64)).cuda()
    occ = torch.ones(nk, nb, dtype=torch.float64, device="cuda")
    plans = [hse.Plan((n, n, n), lattice, kpts, nb, nb, inputs.OMEGA, inputs.ALPHA, dtype=torch.complex64)
             for _ in range(2)]
    ref = hse.hse_fock_apply(plans[0], u, occ, u)
    out = torch.zeros_like(ref)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        hse.hse_fock_apply(plans[1], u, occ, u, out=out)
    # passes that read more blocked arrays leave the graph's copies where they are
    hse.hse_fock_apply_vjp(plans[1], u, occ, u, ref)
    graph.replay()
    assert torch.equal(out, ref)
