"""Plans that work on a smaller grid than the caller's, through the routes around
the plain apply: fixed operator, shards, several streams, deterministic sums, in
cubic and triclinic cells, against the oracle on the caller's grid (1e-10 in FP64
and double-float, 2e-5 and 5e-6 in the mixed form)."""

import numpy as np
import pytest

import oracle
from paper_1305_7313_gb300 import FockPlan, _lib, synth
from tests._common import rel_inf, require_gpu

pytestmark = pytest.mark.gpu

TOL = {_lib.PREC_FP64: (1e-10, 1e-10), _lib.PREC_DF64: (1e-10, 1e-10), _lib.PREC_MIXED32: (2e-5, 5e-6)}
CUBIC = np.eye(3)
TRICLINIC = np.array([[1.0, 0.1, 0.0], [-0.2, 1.0, 0.15], [0.05, -0.1, 1.0]])
# caller's grid, cell, the grid the plan works on (12 Ha)
CASES = [(24, 6.4 * CUBIC, 20), (36, 8.0 * TRICLINIC, 28), (64, 16.0 * TRICLINIC, 56)]


@pytest.mark.parametrize("prec", sorted(TOL), ids=["fp64", "mixed32", "df64"])
@pytest.mark.parametrize("n,cell,work", CASES, ids=[str(c[0]) for c in CASES])
def test_routes_on_a_smaller_working_grid(n, cell, work, prec):
    torch = require_gpu()
    grid = (n,) * 3
    mill, _ = oracle.gsphere(grid, cell, 12.0)
    c = synth.orbitals(mill, cell, 5, n)
    t = synth.orbitals(mill, cell, 3, n + 1)
    occ = np.linspace(2.0, 0.5, 5)
    psi, phi = torch.from_numpy(c).cuda(), torch.from_numpy(t).cuda()
    vr, er, dr = oracle.fock_apply(c, occ, mill, grid, cell, "erfc", 0.3)
    fr = oracle.fock_apply_to(c, occ, t, mill, grid, cell, "erfc", 0.3)
    tv, te = TOL[prec]

    def check(v, e, d):
        assert rel_inf(v.cpu().numpy(), vr) <= tv
        assert abs(e - er) <= te * abs(er) and abs(d - dr) <= te * abs(dr)

    with FockPlan(n, cell, 12.0, _lib.ERFC, 0.3, prec) as plan:
        kept, total = plan.columns()
        assert total == work * 2 * (work // 2 + 1) and 0 < kept <= total
        parts = [plan.apply_shard(psi, occ, s, 3, want_dex=True) for s in range(3)]
        check(sum(p[0] for p in parts), sum(p[1] for p in parts), sum(p[2] for p in parts))
        plan.set_occupied(psi, occ)
        assert rel_inf(plan.apply_fixed(phi).cpu().numpy(), fr) <= tv
        if prec != _lib.PREC_MIXED32:
            plan.set_deterministic(True)
            first = plan.apply(psi, occ, want_dex=True)
            check(*first)
            again = plan.apply(psi, occ, want_dex=True)
            assert torch.equal(first[0], again[0]) and first[1:] == again[1:]
            plan.set_deterministic(False)
        plan.set_batch(1)
        plan.set_streams(3)
        check(*plan.apply(psi, occ, want_dex=True))
