"""The fused FP64 kernel (complex128 grids that fit shared memory) against the FP64 oracle: axes of
every register class, grids whose pencils leave partial warps, several orbitals a CTA, split
partner ranges, fractional and empty occupations, and the exchange energy over an odd and an even
number of orbitals (unordered pairs once; at half the circle of an even number both ends) and over
a down-sampled Fock sum (ordered pairs).  HSE_FP64_FUSED=1 takes the kernel also where a small plan
would choose the staged form.

Tolerance 1e-10, the complex128 bound of the parity tests: eps log2 N per transform and the sums
over partners stay below 1e-12.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1507_05156_gb300 import hse, inputs

pytestmark = pytest.mark.gpu

# grid, nk, n_occ, n_tgt, kocc
CASES = [((2, 3, 5), 1, 1, 1, None), ((5, 4, 6), 3, 3, 17, None), ((12, 10, 9), 2, 3, 2, None), ((12, 12, 12), 2, 4, 3, None),
         ((16, 15, 4), 2, 2, 3, None), ((16, 16, 16), 1, 5, 2, None), ((18, 4, 20), 2, 2, 1, None), ((24, 6, 8), 1, 3, 2, None),
         ((25, 2, 3), 2, 2, 5, None), ((4, 32, 10), 1, 2, 2, None), ((8, 8, 8), 4, 3, 5, (1, 3)), ((9, 8, 5), 3, 2, 2, (2,))]


@pytest.mark.parametrize("grid,nk,n_occ,n_tgt,kocc", CASES)
def test_fused_f64(grid, nk, n_occ, n_tgt, kocc, monkeypatch):
    monkeypatch.setenv("HSE_FP64_FUSED", "1")
    lattice = np.array([[7.1, 0.3, -0.4], [0.9, 6.2, 0.5], [-0.6, 1.1, 5.3]])
    rng = np.random.default_rng(sum(grid) + 100 * nk + n_tgt)
    kpts = (rng.random((nk, 3)) - 0.5) @ (2 * np.pi * np.linalg.inv(lattice).T)
    u_occ, u_tgt = (inputs.random_orbitals(s, (nk, n) + grid) * 0.1 for s, n in ((nk + 1, n_occ), (nk + 2, n_tgt)))
    ybar = inputs.random_orbitals(nk + 3, u_tgt.shape) * 0.1
    occ = rng.random((nk, n_occ))
    if n_occ > 1:
        occ[0, 0] = 0.0
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    rel = lambda a, b: np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b)  # noqa: E731
    ks = None if kocc is None else list(kocc)
    plan = hse.Plan(grid, lattice, kpts, n_occ, n_tgt, 0.2, 0.25, dtype=torch.complex128, kocc=ks)
    kw = {} if ks is None else {"kocc": ks}
    out = hse.hse_fock_apply(plan, dev(u_occ), dev(occ), dev(u_tgt))
    assert rel(out, oracle.fock_apply(u_occ, occ, u_tgt, kpts, lattice, grid, 0.2, 0.25, **kw)) <= 1e-10
    e = hse.hse_exchange_energy(plan, dev(u_occ), dev(occ)).item()
    e_ref = oracle.exchange_energy(u_occ, occ, kpts, lattice, grid, 0.2, 0.25, 2.0, **kw)
    assert abs(e - e_ref) <= 1e-10 * abs(e_ref)
    g_occ, g_tgt, g_om = hse.hse_fock_apply_vjp(plan, dev(u_occ), dev(occ), dev(u_tgt), dev(ybar))
    r_occ, r_tgt, r_om = oracle.fock_apply_vjp(u_occ, occ, u_tgt, ybar, kpts, lattice, grid, 0.2, 0.25, **kw)
    assert rel(g_occ, r_occ) <= 1e-10 and rel(g_tgt, r_tgt) <= 1e-10
    assert abs(g_om.item() - r_om) <= 1e-10 * abs(r_om)
    hse.hse_status(plan)
