"""Tilings of the pair passes: what a plan reports is of the grid its passes run on,
every index a grid size had is taken, and each gives the oracle's results (1e-10 in
FP64, 2e-5 and 5e-6 in the mixed form)."""

import itertools

import numpy as np
import pytest

import oracle
from paper_1305_7313_gb300 import FockPlan, _lib, synth
from tests._common import cubic, rel_inf, require_gpu

pytestmark = pytest.mark.gpu

TOL = {_lib.PREC_FP64: (1e-10, 1e-10), _lib.PREC_MIXED32: (2e-5, 5e-6)}
FORMS = pytest.mark.parametrize("prec", sorted(TOL), ids=["fp64", "mixed32"])


def product(tiling):
    return int(np.prod(tiling["radices"]))


@FORMS
def test_both_tilings_of_16_give_the_oracles_results(prec):
    torch = require_gpu()
    n, cell = 16, cubic(4.8)
    mill, _ = oracle.gsphere((n,) * 3, cell, 8.0)
    c, occ = synth.orbitals(mill, cell, 5, 3), np.linspace(2.0, 1.0, 5)
    vr, er, dr = oracle.fock_apply(c, occ, mill, (n,) * 3, cell, "erfc", 0.3)
    tv, te = TOL[prec]
    with FockPlan(n, cell, 8.0, _lib.ERFC, 0.3, prec) as plan:
        assert plan.columns()[1] == n * 2 * (n // 2 + 1)  # works on 16^3 itself
        for passes in plan.tilings().values():
            assert len(passes) == 2 and all(product(t) == n for t in passes)
            assert passes[0] != passes[1]
        for tiles in itertools.product((0, 1), repeat=3):
            plan.set_tiling(tiles)
            v, e, d = plan.apply(torch.from_numpy(c).cuda(), occ, want_dex=True)
            assert rel_inf(v.cpu().numpy(), vr) <= tv
            assert abs(e - er) <= te * abs(er) and abs(d - dr) <= te * abs(dr)
