"""The bounded waits of the two-exchange 16^3 kernels, without a GPU fault: plans created with
HSE_INJECT_SKIP_FILL=1 never issue their first partner copies, so the waits run out (about a second
each).  The kernels have to record HSE_ERR_TIMEOUT, finish, and leave the context usable.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1507_05156_gb300 import hse, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["apply", "u_occ", "u_occ and omega"])
def test_two_exchange_kernels_report_timeout(call, monkeypatch):
    c = inputs.make_cell(78, (16, 16, 16), (1, 1, 1), 3)  # one work item
    u = torch.from_numpy(c.u_occ.astype(np.complex64)).cuda()
    occ = torch.from_numpy(c.occ).cuda()

    def run(plan):
        if call == "apply":
            return hse.hse_fock_apply(plan, u, occ, u)
        return hse.hse_fock_apply_vjp(plan, u, occ, u, u.conj().resolve_conj().contiguous(), need_tgt=False,
                                      need_omega=call != "u_occ")[0]

    make = lambda: hse.Plan(c.grid, c.lattice, c.kpts, c.n_occ, c.n_tgt, c.omega, c.alpha)  # noqa: E731
    monkeypatch.setenv("HSE_BLOCKS_PER_SM", "6")
    monkeypatch.setenv("HSE_RANGES", "1")
    monkeypatch.setenv("HSE_INJECT_SKIP_FILL", "1")
    bad = make()
    monkeypatch.delenv("HSE_INJECT_SKIP_FILL")
    run(bad)
    with pytest.raises(hse.HseError) as ei:
        hse.hse_status(bad)
    assert ei.value.code == -5  # HSE_ERR_TIMEOUT
    hse.hse_status(bad)  # the status word was cleared
    good = make()
    got = run(good).cpu().numpy()
    hse.hse_status(good)
    w = c.u_occ.astype(np.complex64).astype(np.complex128)
    args = (c.kpts, c.lattice, c.grid, c.omega, c.alpha)
    ref = oracle.fock_apply(w, c.occ, w, *args) if call == "apply" else oracle.fock_apply_vjp(w, c.occ, w, w.conj(), *args)[0]
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)
