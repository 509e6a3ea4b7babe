"""Scratch of the orthonormalisation over orders of calls: after more bands than the tiled kernels
take, around a captured graph, where its allocation fails, and with complex128 calls that overlap on
two streams.  References: the FP64 oracle (complex64 within 1e-6, one FP32 rounding; complex128
within 1e-12), and for the overlapping calls the same calls one after the other.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1507_05156_gb300 import hse, inputs

pytestmark = pytest.mark.gpu

N, NK = 8, 3


def _plan(nk=NK, dtype=torch.complex64):
    lattice = inputs.cubic_lattice(inputs.A_SI)
    kpts = np.arange(3.0 * nk).reshape(nk, 3) * 0.01
    return hse.Plan((N,) * 3, lattice, kpts, 1, 1, 0.2, 0.25, dtype=dtype), abs(np.linalg.det(lattice)) / N ** 3


def _u(nb, seed, nk=NK, dtype=np.complex64):
    return (inputs.random_orbitals(seed, (nk, nb) + (N,) * 3) * 0.05).astype(dtype)


def _check(got, u, dV, tol):
    q = oracle.ortho.gram_schmidt(u.astype(np.complex128), dV)
    nb = u.shape[0] * u.shape[1]
    err = np.linalg.norm((got.cpu().numpy() - q).reshape(nb, -1), axis=1) / np.linalg.norm(q.reshape(nb, -1), axis=1)
    assert err.max() <= tol


@pytest.mark.parametrize("between", [(), (8,)])
def test_graph_after_many_bands(between):
    """80 bands (no factors), a graph of 8, 32 bands outside it, a replay: nothing the graph uses moves,
    and nothing is allocated while it is captured."""
    plan, dV = _plan()
    for nb in (80,) + between:
        hse.hse_orthonormalize(plan, torch.from_numpy(_u(nb, nb)).cuda())
    u = _u(8, 1)
    d = torch.from_numpy(u).cuda()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        hse.hse_orthonormalize(plan, d)
    more = _u(32, 2)
    dm = torch.from_numpy(more).cuda()
    hse.hse_orthonormalize(plan, dm)
    _check(dm, more, dV, 1e-6)
    d.copy_(torch.from_numpy(u))
    graph.replay()
    hse.hse_status(plan)
    _check(d, u, dV, 1e-6)


@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
def test_scratch_allocation_fails(dtype, monkeypatch):
    """Without memory for the factors Gram-Schmidt does the call, and a graph can still be captured."""
    npdt = np.complex64 if dtype == torch.complex64 else np.complex128
    tol = 1e-6 if dtype == torch.complex64 else 1e-12
    monkeypatch.setenv("HSE_BLOCKS_PER_SM", "-1")
    monkeypatch.setenv("HSE_FP64_FUSED", "0")
    for k in range(100):  # the plan's own allocations, none of which it can do without
        monkeypatch.setenv("HSE_FAIL_ALLOC_AT", str(k))
        try:
            _plan(dtype=dtype)
            break
        except hse.HseError:
            pass
    monkeypatch.setenv("HSE_FAIL_ALLOC_AT", str(k + (1 if dtype == torch.complex64 else 0)))
    plan, dV = _plan(dtype=dtype)
    u = _u(12, 5, dtype=npdt)
    d = torch.from_numpy(u).cuda()
    hse.hse_orthonormalize(plan, d)
    hse.hse_status(plan)
    _check(d, u, dV, tol)
    d.copy_(torch.from_numpy(u))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        hse.hse_orthonormalize(plan, d)
    graph.replay()
    hse.hse_status(plan)
    _check(d, u, dV, tol)


def test_complex128_calls_overlap_on_two_streams():
    nk, nb = 96, 24
    plan, _ = _plan(nk, torch.complex128)
    us = [torch.from_numpy(_u(nb, s, nk, np.complex128)).cuda() for s in (3, 4)]
    ref = [hse.hse_orthonormalize(plan, u.clone()) for u in us]
    streams = [torch.cuda.Stream() for _ in us]
    torch.cuda.synchronize()
    for _ in range(4):
        out = [u.clone() for u in us]
        torch.cuda.synchronize()
        for s, o in zip(streams, out):
            hse.hse_orthonormalize(plan, o, stream=s)
        torch.cuda.synchronize()
        for o, r in zip(out, ref):
            assert torch.linalg.vector_norm(o - r) <= 1e-12 * torch.linalg.vector_norm(r)
