"""Calls as the first CUDA work of a host thread that has no context yet (an autograd thread with a
cotangent already made): every pass whose kernel reads its partners through a tensor map.  The thread
calls the C entry points on arrays made elsewhere, so nothing else binds a context before them; the
result has to be the one that the main thread gets.
"""
import threading

import numpy as np
import pytest
import torch

from paper_1507_05156_gb300 import hse, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,variant,call", [(12, -1, "apply"), (16, 6, "apply"), (16, 6, "u_occ"), (12, -1, "omega"),
                                            (18, -1, "energy")])
def test_first_cuda_work_of_a_thread(n, variant, call, monkeypatch):
    monkeypatch.setenv("HSE_BLOCKS_PER_SM", str(variant))
    nb, grid = 2, (n, n, n)
    plan = hse.Plan(grid, inputs.cubic_lattice(inputs.A_SI), np.zeros((1, 3)), nb, nb, inputs.OMEGA, inputs.ALPHA)
    u = torch.from_numpy(inputs.random_orbitals(n, (1, nb) + grid).astype(np.complex64)).cuda()
    y = u.conj().resolve_conj().contiguous()
    occ = torch.ones(1, nb, dtype=torch.float64, device="cuda")
    lib, stream = hse.load_library(), hse._stream()

    def run(out, val):
        a = [hse._ptr(t) for t in (u, occ, u, y, out)] + [hse._ptr(val)]
        if call == "apply":
            return lib.hse_fock_apply(plan.handle, a[0], a[1], a[2], a[4], stream)
        if call == "energy":
            return lib.hse_exchange_energy(plan.handle, a[0], a[1], a[5], stream)
        return lib.hse_fock_apply_vjp(plan.handle, *a[:4], a[4] if call == "u_occ" else None, None,
                                      a[5] if call == "omega" else None, stream)

    outs = [(torch.zeros_like(u), torch.zeros((), dtype=torch.float64, device="cuda")) for _ in range(2)]
    codes = []
    t = threading.Thread(target=lambda: codes.append(run(*outs[0])))
    torch.cuda.synchronize()
    t.start()
    t.join()
    assert codes == [0]
    assert run(*outs[1]) == 0
    hse.hse_status(plan)
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
    assert outs[1][0].abs().sum() > 0 or outs[1][1] != 0
