"""Shards of an apply, more of them than there are chains: the ones without pairs
give zeros, and all of them add up to the full apply (to the order of the sums:
1e-13, as for other shard counts; the mixed form to its own bounds)."""

import numpy as np
import pytest

import oracle
from paper_1305_7313_gb300 import FockPlan, _lib, synth
from tests._common import cubic, rel_inf, require_gpu

pytestmark = pytest.mark.gpu

TOL = {_lib.PREC_FP64: (1e-13, 1e-13), _lib.PREC_DF64: (1e-13, 1e-13), _lib.PREC_MIXED32: (2e-5, 5e-6)}


# (deterministic accumulation is not offered for the mixed form)
FORMS = {"fp64": (_lib.PREC_FP64, False), "mixed32": (_lib.PREC_MIXED32, False), "df64": (_lib.PREC_DF64, False),
         "fp64-det": (_lib.PREC_FP64, True), "df64-det": (_lib.PREC_DF64, True)}


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("nb", [1, 2, 3])
def test_shards_without_pairs(nb, form):
    torch = require_gpu()
    prec, det = FORMS[form]
    n, cell, nshards = 24, cubic(10.0), 8
    mill, _ = oracle.gsphere((n,) * 3, cell, 10.0)
    psi = torch.from_numpy(synth.orbitals(mill, cell, nb, nb)).cuda()
    occ = np.array([2.0, 1.5, 1.0])[:nb]
    with FockPlan(n, cell, 10.0, _lib.ERFC, 0.3, prec) as plan:
        plan.set_deterministic(det)
        full, efull, dfull = plan.apply(psi, occ, want_dex=True)
        total, esum, dsum, empty = torch.zeros_like(full), 0.0, 0.0, 0
        for s in range(nshards):
            v = torch.full_like(psi, complex(np.nan, np.nan))
            v, e, d = plan.apply_shard(psi, occ, s, nshards, v, want_dex=True)
            if len(_lib.fock_schedule(nb, s, nshards)) == 0:
                empty += 1
                assert e == 0.0 and d == 0.0 and bool(torch.all(v == 0).item())
            total, esum, dsum = total + v, esum + e, dsum + d
    assert empty == nshards - (nb * (nb + 1) // 2 + 1) // 2
    tv, te = TOL[prec]
    assert rel_inf(total.cpu().numpy(), full.cpu().numpy()) <= tv
    assert abs(esum - efull) <= te * abs(efull) and abs(dsum - dfull) <= te * abs(dfull)
