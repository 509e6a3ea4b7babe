"""Plans where memory is short: what a plan can do without does not fail its creation (the copies of the
two-CTA apply, the ranges of the fused FP64 passes), and a batched plan holds no copies that its form
may never read.  HSE_FAIL_ALLOC_AT=k fails the plan's k-th allocation as an exhausted device would.
Tolerances are those of the parity tests.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1507_05156_gb300 import hse, inputs

pytestmark = pytest.mark.gpu


def _apply(plan, c, u, occ):
    before = hse.kernel_launches()
    out = hse.hse_fock_apply(plan, u, occ, u)
    hse.hse_status(plan)
    return out, hse.kernel_launches() - before


@pytest.mark.parametrize("n,dtype,env,fewer", [(12, torch.complex64, ("HSE_BLOCKS_PER_SM", "7"), 1),
                                               (20, torch.complex64, ("HSE_BLOCKS_PER_SM", "7"), 1),
                                               (12, torch.complex128, ("HSE_FP64_FUSED", "1"), 1)])
def test_creation_does_without(n, dtype, env, fewer, monkeypatch):
    """The first allocation whose failure leaves a plan is the dispensable one: the plan then computes
    with fewer launches (no blocked copy; no sum of ranges)."""
    monkeypatch.setenv(*env)
    c = inputs.make_cell(inputs.SEED_BASE + 320, (n, n, n), (2, 1, 1), 3)
    make = lambda: hse.Plan(c.grid, c.lattice, c.kpts, c.n_occ, c.n_tgt, c.omega, c.alpha, dtype=dtype)  # noqa: E731
    npdt = np.complex64 if dtype == torch.complex64 else np.complex128
    u_h = c.u_occ.astype(npdt)
    u, occ = torch.from_numpy(u_h).cuda(), torch.from_numpy(c.occ).cuda()
    _, launches = _apply(make(), c, u, occ)
    for k in range(100):
        monkeypatch.setenv("HSE_FAIL_ALLOC_AT", str(k))
        try:
            plan = make()
            break
        except hse.HseError as e:
            assert e.code == -6
    out, got = _apply(plan, c, u, occ)
    assert got == launches - fewer
    w = u_h.astype(np.complex128)
    ref = oracle.fock_apply(w, c.occ, w, c.kpts, c.lattice, c.grid, c.omega, c.alpha)
    tol = 1e-5 if dtype == torch.complex64 else 1e-10
    assert np.linalg.norm(out.cpu().numpy() - ref) <= tol * np.linalg.norm(ref)
    y = u.conj().resolve_conj().contiguous()
    g = hse.hse_fock_apply_vjp(plan, u, occ, u, y)
    hse.hse_status(plan)
    r = oracle.fock_apply_vjp(w, c.occ, w, w.conj(), c.kpts, c.lattice, c.grid, c.omega, c.alpha)
    assert np.linalg.norm(g[0].cpu().numpy() - r[0]) <= tol * np.linalg.norm(r[0])


def test_batched_plan_holds_no_copies(monkeypatch):
    """A batched plan of cells whose single-cell apply is the two-CTA one takes no more memory with the
    pencil-blocked copies than without."""
    monkeypatch.setenv("HSE_BLOCKS_PER_SM", "7")
    c = inputs.make_cell(inputs.SEED_BASE + 321, (18, 18, 18), (3, 3, 3), 12)
    free = lambda: (torch.cuda.synchronize(), torch.cuda.mem_get_info()[0])[1]  # noqa: E731
    used = []
    for blocks in ("1", "0", "1"):  # the first plan of a process loads the kernels too
        monkeypatch.setenv("HSE_PENCIL_BLOCKS", blocks)
        f0 = free()
        plan = hse.BatchedPlan([c])
        used.append(f0 - free())
        del plan
    copies = 3 * 27 * 12 * 18 ** 3 * 8
    assert used[2] <= used[1] + copies // 2
