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


@FORMS
def test_a_plan_on_a_smaller_grid_reports_the_tilings_it_runs(prec):
    # 96^3 at L 24: the pair passes run on 80^3, which has one tiling; index 1, which
    # 96^3 has, is still taken, and those passes run the one there is
    torch = require_gpu()
    n, cell = 96, cubic(24.0)
    with FockPlan(n, cell, 12.0, precision=prec) as plan:
        assert plan.columns()[1] == 80 * 2 * 41
        for p, name in enumerate(_lib.PASSES):
            (tiling,) = plan.tilings()[name]
            assert product(tiling) == 80
            with pytest.raises(_lib.FockError):
                _lib.fock_plan_tiling_info(plan.handle, p, 1)
        psi = torch.from_numpy(synth.orbitals(plan.miller, cell, 2, 5)).cuda()
        occ = np.array([2.0, 1.0])
        v0, e0, _ = plan.apply(psi, occ)
        plan.set_tiling([1, 1, 1])
        v1, e1, _ = plan.apply(psi, occ)
        tv, te = TOL[prec]
        assert rel_inf(v1.cpu().numpy(), v0.cpu().numpy()) <= tv and abs(e1 - e0) <= te * abs(e0)
        for bad in ([2, 0, 0], [0, -1, 0]):
            with pytest.raises(_lib.FockError):
                plan.set_tiling(bad)
    with FockPlan(48, cubic(13.5), 12.0, precision=prec) as plan:  # 48 has one
        with pytest.raises(_lib.FockError):
            plan.set_tiling([1, 0, 0])
