"""The fixed operator on a stream of its own, its work still queued when the next
call grows the plan's workspace (1e-10 and 2e-5 against the oracle, as elsewhere)."""

import numpy as np
import pytest

import oracle
from paper_1305_7313_gb300 import FockBatch, FockPlan, _lib, synth
from tests._common import cubic, rel_inf, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [(_lib.PREC_FP64, 1e-10), (_lib.PREC_DF64, 1e-10), (_lib.PREC_MIXED32, 2e-5)],
                         ids=["fp64", "df64", "mixed32"])
def test_growing_waits_for_the_occupied_set(prec, tol):
    torch = require_gpu()
    n, cell = 24, cubic(9.0)
    with FockPlan(n, cell, 8.0, _lib.ERFC, 0.4, prec) as plan:
        c, t = synth.orbitals(plan.miller, cell, 5, 1), synth.orbitals(plan.miller, cell, 4, 2)
        occ = np.array([2.0, 1.5, 1.0, 0.5, 0.25])
        psi, phi = torch.from_numpy(c).cuda(), torch.from_numpy(t).cuda()
        torch.cuda.synchronize()
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            torch.cuda._sleep(20_000_000)  # about 10 ms
            plan.set_occupied(psi, occ)
            v = plan.apply_fixed(phi)  # room for 9 bands instead of 5
        s.synchronize()
        vr = oracle.fock_apply_to(c, occ, t, plan.miller, (n,) * 3, cell, "erfc", 0.4)
        assert rel_inf(v.cpu().numpy(), vr) <= tol


def test_a_batch_drops_the_occupied_set():
    # a batch takes the plan's workspace over: the operator fixed before is gone
    torch = require_gpu()
    n, cell = 24, cubic(9.0)
    with FockPlan(n, cell, 8.0, _lib.ERFC, 0.4) as plan:
        psi = torch.from_numpy(synth.orbitals(plan.miller, cell, 5, 1)).cuda()
        occ = np.full(5, 2.0)
        plan.set_occupied(psi, occ)
        before = plan.apply_fixed(psi)
        b = FockBatch([plan], [psi[:3].contiguous()], [occ[:3]])
        b.run()
        b.close()
        with pytest.raises(_lib.FockError):
            plan.apply_fixed(psi)
        plan.set_occupied(psi, occ)
        assert rel_inf(plan.apply_fixed(psi).cpu().numpy(), before.cpu().numpy()) <= 1e-12
