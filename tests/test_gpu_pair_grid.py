"""Plans whose working grid is smaller than the caller's (and the sizes compiled
for them alone) against the oracle on the caller's grid, with the tolerances of
the parity tests (1e-10 for FP64 and double-float, 2e-5 and 5e-6 for the mixed
form); every entry that takes a grid of the caller's size still does."""

import numpy as np
import pytest

import oracle
from oracle.sternheimer import sternheimer_solve
from paper_1305_7313_gb300 import FockBatch, FockKPlan, FockPlan, _lib, synth
from tests._common import cubic, rel_inf, require_gpu

pytestmark = pytest.mark.gpu

TOL = {_lib.PREC_FP64: (1e-10, 1e-10), _lib.PREC_DF64: (1e-10, 1e-10), _lib.PREC_MIXED32: (2e-5, 5e-6)}
# caller's grid and cell edge at 12 Ha -> working grid 20, 28, 32, 40, 56, 60, 64, 80
CASES = [(24, 6.4), (32, 8.5), (36, 10.125), (48, 12.5), (64, 17.0), (64, 18.0), (72, 20.0), (96, 24.0)]


@pytest.mark.parametrize("prec", sorted(TOL), ids=["fp64", "mixed32", "df64"])
@pytest.mark.parametrize("n,length", CASES)
def test_apply_matches_the_oracle_on_the_callers_grid(n, length, prec):
    torch = require_gpu()
    cell = cubic(length)
    mill, _ = oracle.gsphere((n, n, n), cell, 12.0)
    c = synth.orbitals(mill, cell, 3, n)
    occ = np.array([2.0, 1.25, 0.5])
    with FockPlan(n, cell, 12.0, _lib.ERFC, 0.3, prec) as plan:
        v, e, d = plan.apply(torch.from_numpy(c).cuda(), occ, want_dex=True)
        v = v.cpu().numpy()
    vr, er, dr = oracle.fock_apply(c, occ, mill, (n, n, n), cell, "erfc", 0.3)
    tv, te = TOL[prec]
    assert rel_inf(v, vr) <= tv and abs(e - er) <= te * abs(er) and abs(d - dr) <= te * abs(dr)


def test_pair_energies_and_the_static_entry():
    torch = require_gpu()
    n, cell = 24, cubic(6.4)
    with FockPlan(n, cell, 12.0) as plan:
        psi = torch.from_numpy(synth.orbitals(plan.miller, cell, 4, 5)).cuda()
        pairs = [(0, 0), (1, 3), (2, 1)]
        e, _ = plan.pair_energies(psi, pairs, want_d=True)
        es, _ = _lib.fock_pair_energies_static(plan.handle, psi, pairs, want_d=True)
        np.testing.assert_allclose(es, e, rtol=1e-12)
        r = oracle.orbitals_to_real(psi.cpu().numpy(), plan.miller, (n,) * 3, cell, real=True)
        from oracle.fock import kernel_grid
        vg, dvg = kernel_grid("spencer_alavi", (n,) * 3, cell, None)
        for k, (i, j) in enumerate(pairs):
            assert abs(e[k] - oracle.pair_energy(r[i], r[j], vg, dvg)[0]) <= 1e-10 * abs(e[k])


@pytest.mark.parametrize("prec", [_lib.PREC_FP64, _lib.PREC_MIXED32], ids=["fp64", "mixed32"])
def test_k_points_match_the_oracle_on_the_callers_grid(prec):
    torch = require_gpu()
    n, cell = 32, cubic(7.9)  # working grid 28
    kpts, wk = np.array([[0.0, 0.0, 0.0], [0.5, 0.0, 0.0], [0.25, -0.25, 0.5]]), np.array([0.5, 0.3, 0.2])
    plan = FockKPlan(n, cell, 12.0, kpts, wk, _lib.ERFC, 0.4, prec)
    c = [synth.orbitals_k(plan.miller(k), cell, kpts[k], 2, 60 + k) for k in range(3)]
    occ = np.array([[2.0, 1.0]] * 3)
    v, e = plan.apply([torch.from_numpy(x).cuda() for x in c], occ)
    vr, er = oracle.fock_apply_kpoints(c, occ, [plan.miller(k) for k in range(3)], kpts, wk, (n,) * 3, cell, "erfc", 0.4)
    tv, te = TOL[prec]
    vmax = max(np.max(np.abs(x)) for x in vr)
    assert abs(e - er) <= te * abs(er)
    for a, b in zip(v, vr):
        assert np.max(np.abs(a.cpu().numpy() - b)) <= tv * vmax
    plan.close()


@pytest.mark.parametrize("prec", [_lib.PREC_FP64, _lib.PREC_MIXED32], ids=["fp64", "mixed32"])
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_batches_of_such_plans_match_single_applies(mode, prec):
    torch = require_gpu()
    plans, psi, occ = [], [], []
    for n, length in CASES:
        if n == 36:
            continue  # not a batch size
        cell = cubic(length)
        p = FockPlan(n, cell, 12.0, _lib.SPENCER_ALAVI, None, prec)
        plans.append(p)
        psi.append(torch.from_numpy(synth.orbitals(p.miller, cell, 3, n)).cuda())
        occ.append(np.array([2.0, 1.0, 0.5]))
    b = FockBatch(plans, psi, occ, persistent=mode)
    ex, _ = b.run()
    got = [x.clone() for x in b.vpsi]
    b.close()
    tv, te = TOL[prec]
    for k, p in enumerate(plans):
        v, e, _ = p.apply(psi[k], occ[k])
        assert abs(ex[k] - e) <= te * abs(e)
        assert rel_inf(got[k].cpu().numpy(), v.cpu().numpy()) <= tv
        p.close()


def test_sternheimer_takes_its_potential_on_the_callers_grid():
    # the potential has components beyond the working grid (20^3); chain batch 1,
    # so the plan's transform buffer is smaller than one block of the caller's grid
    torch = require_gpu()
    n, cell = 24, cubic(6.4)
    with FockPlan(n, cell, 12.0) as plan:
        plan.set_batch(1)
        rng = np.random.default_rng(4)
        v = rng.standard_normal((n, n, n))
        u = synth.orbitals(plan.miller, cell, 3, 1)
        w = synth.orbitals(plan.miller, cell, 5, 2)
        eps = v.min() - 2.0 - 0.1 * np.arange(5)
        g, it, res = plan.sternheimer(torch.from_numpy(v).cuda(), torch.from_numpy(u).cuda(), eps,
                                      torch.from_numpy(w).cuda(), 1.0, 1e-10)
        g = g.cpu().numpy()
        # each oracle system has its own eps; same CG, so the same iterates
        go, ito, _ = sternheimer_solve(u, eps, w, v, plan.miller, (n,) * 3, cell, 1.0, 1e-10)
        assert np.all(np.abs(it - ito) <= 2 + 0.05 * ito)
        assert rel_inf(g, go) <= 1e-8
        # the plan still applies
        c = torch.from_numpy(u).cuda()
        vx, ex, _ = plan.apply(c, np.full(3, 2.0))
        vr, er, _ = oracle.fock_apply(u, np.full(3, 2.0), plan.miller, (n,) * 3, cell, "spencer_alavi")
        assert rel_inf(vx.cpu().numpy(), vr) <= 1e-10 and abs(ex - er) <= 1e-10 * abs(er)


@pytest.mark.parametrize("nb", [1, 15, 16, 17, 32, 33, 48, 49, 64, 65, 97])
def test_overlaps_of_every_tile_size(nb):
    # constant orbitals: only the G = 0 term is left, which the mixed form takes
    # from the FP64 overlaps, so that a missed entry of a tile shows in E_x; a
    # second call with other occupations, its energy not asked for, comes between
    torch = require_gpu()
    e = {}
    for prec in (_lib.PREC_FP64, _lib.PREC_MIXED32):
        with FockPlan(16, cubic(5.5), 6.0, precision=prec) as plan:
            c = np.zeros((nb, plan.npw), dtype=np.complex128)
            c[:, int(np.flatnonzero(np.all(plan.miller == 0, axis=1))[0])] = 1.0 + np.arange(nb) / nb
            psi, v = torch.from_numpy(c).cuda(), torch.empty((nb, plan.npw), dtype=torch.complex128, device="cuda")
            occ = 2.0 - np.arange(nb) / nb
            first = _lib.fock_apply(plan.handle, psi, occ, v)[0]
            _lib.fock_apply(plan.handle, psi, np.ones(nb), v, want_ex=False)
            e[prec] = _lib.fock_apply(plan.handle, psi, occ, v)[0]
            assert abs(first - e[prec]) <= 1e-13 * abs(first)
    assert abs(e[_lib.PREC_MIXED32] - e[_lib.PREC_FP64]) <= 1e-12 * abs(e[_lib.PREC_FP64])
