"""The omega gradient of the two-exchange 16^3 kernel sums at most 16 products in FP32 before they go
to FP64.

One k-point, a constant occupied orbital, and targets that hold three plane waves along the first axis,
m = 4, 12 (= -4) and 8, so that every transform is exact in FP32: A = (L, L, s), B = (L', -L', s').  The
terms of m = +-4 cancel exactly, and what is left, dv(8) s s', is 2^-20 of them.  A thread holds m = 0,
4, 8, 12: with all its products in one FP32 sum the result is wrong in its second digit.  Bound: the
roundings of dv, of its product and of the two scale factors, 5 x 2^-24 = 3e-7; 1e-6 is asked for.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1507_05156_gb300 import hse

pytestmark = pytest.mark.gpu


def test_cancelling_products(monkeypatch):
    monkeypatch.setenv("HSE_BLOCKS_PER_SM", "6")
    n, omega, alpha = 16, 0.2, 0.25
    grid, lattice, kpts = (n,) * 3, np.eye(3) * 200.0, np.zeros((1, 3))
    x = np.arange(n).reshape(n, 1, 1) * np.ones(grid)
    s = 2.0 ** -10
    quarter = lambda f: np.round(f(np.pi * x / 2.0))  # noqa: E731
    u_i = 2.0 * quarter(np.cos) + s * quarter(lambda a: np.cos(2.0 * a))
    ybar = 2.0j * quarter(np.sin) + s * quarter(lambda a: np.cos(2.0 * a))
    u_j = np.full(grid, 0.25)
    c64 = lambda a: np.ascontiguousarray(a[None, None]).astype(np.complex64)  # noqa: E731
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    occ = np.ones((1, 1))
    plan = hse.Plan(grid, lattice, kpts, 1, 1, omega, alpha)
    _, _, g = hse.hse_fock_apply_vjp(plan, dev(c64(u_j)), dev(occ), dev(c64(u_i)), dev(c64(ybar)), need_tgt=False)
    hse.hse_status(plan)
    w = [c64(a).astype(np.complex128) for a in (u_j, u_i, ybar)]
    ref = oracle.fock_apply_vjp(w[0], occ, w[1], w[2], kpts, lattice, grid, omega, alpha)[2]
    m8 = 8 * 2 * np.pi / 200.0  # the closed form, so that the reference's own cancellation does not count
    dv = -2.0 * np.pi / omega ** 3 * np.exp(-(m8 / (2.0 * omega)) ** 2)
    closed = -alpha * dv * (0.25 * s) ** 2 * n ** 3
    assert abs(ref - closed) <= 1e-8 * abs(closed)
    assert abs(g.item() - closed) <= 1e-6 * abs(closed)
