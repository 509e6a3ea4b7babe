"""The tiled Gram kernel and the Cholesky orthonormalisation at their edges, against the FP64 oracle:
band counts around the 4-band tiles, the 10-tile groups and the 64-band limit, grids that are no
multiple of a run of points, and k-points whose bands are nearly dependent (which take the
modified Gram-Schmidt kernel) beside well-conditioned ones.

Tolerances: overlaps 1e-12 of the largest (FP64 sums of up to 4096 terms); orthonormal bands 1e-12
(complex128) and 1e-6 (complex64, one FP32 rounding), times the condition number (1e4) for the nearly
dependent set.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1507_05156_gb300 import hse, inputs

pytestmark = pytest.mark.gpu


def _plan(grid, nk, nb, dtype):
    lattice = inputs.cubic_lattice(inputs.A_SI)
    kpts = np.arange(3.0 * nk).reshape(nk, 3) * 0.01
    return hse.Plan(grid, lattice, kpts, 1, 1, 0.2, 0.25, dtype=dtype), abs(np.linalg.det(lattice)) / np.prod(grid)


@pytest.mark.parametrize("n,nk,nb,dtype", [(4, 1, 1, torch.complex64), (6, 2, 3, torch.complex64), (6, 3, 4, torch.complex128),
                                           (10, 2, 9, torch.complex64), (12, 1, 17, torch.complex128),
                                           (16, 1, 64, torch.complex64), (16, 1, 65, torch.complex64),
                                           (12, 2, 40, torch.complex128)])
def test_overlap_and_orthonormalize(n, nk, nb, dtype):
    grid = (n, n, n)
    plan, dV = _plan(grid, nk, nb, dtype)
    u = inputs.random_orbitals(nb, (nk, nb) + grid) * 0.05
    npdt = np.complex64 if dtype == torch.complex64 else np.complex128
    u = u.astype(npdt)
    cond = 1.0
    if nb >= 3:  # the last k-point: band 2 within 1e-4 of the span of the first two
        u[-1, 2] = ((0.5 - 0.25j) * u[-1, 0] + 2.0 * u[-1, 1] + 1e-4 * u[-1, 2]).astype(npdt)
        cond = 1e4
    d = torch.from_numpy(u).cuda()
    w = u.astype(np.complex128)
    S = hse.hse_overlap(plan, d).cpu().numpy()
    ref = oracle.ortho.overlap(w, dV)
    assert np.abs(S - ref).max() <= 1e-12 * np.abs(ref).max()
    assert np.abs(S - np.conj(np.transpose(S, (0, 2, 1)))).max() == 0.0
    hse.hse_orthonormalize(plan, d)
    hse.hse_status(plan)
    q = oracle.ortho.gram_schmidt(w, dV)
    got = d.cpu().numpy().astype(np.complex128)
    tol = 1e-12 if dtype == torch.complex128 else 1e-6
    for k in range(nk):
        err = np.linalg.norm((got[k] - q[k]).reshape(nb, -1), axis=1) / np.linalg.norm(q[k].reshape(nb, -1), axis=1)
        assert err.max() <= tol * (cond if k == nk - 1 else 1.0)


def test_first_complex128_call_is_captured():
    """A plan's first complex128 call, captured into a graph, allocates nothing; a call with more bands
    in between does not disturb its replay."""
    n, nk, nb = 12, 2, 6
    plan, dV = _plan((n, n, n), nk, nb, torch.complex128)
    u = inputs.random_orbitals(7, (nk, nb, n, n, n)) * 0.05
    d = torch.from_numpy(u).cuda()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        hse.hse_orthonormalize(plan, d)
    big = torch.from_numpy(inputs.random_orbitals(8, (nk, 2 * nb, n, n, n)) * 0.05).cuda()
    hse.hse_orthonormalize(plan, big)
    d.copy_(torch.from_numpy(u))
    graph.replay()
    hse.hse_status(plan)
    q = oracle.ortho.gram_schmidt(u, dV)
    err = np.linalg.norm((d.cpu().numpy() - q).reshape(nk * nb, -1), axis=1) / np.linalg.norm(q.reshape(nk * nb, -1), axis=1)
    assert err.max() <= 1e-12
