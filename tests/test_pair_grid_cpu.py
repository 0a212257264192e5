"""The plans' working grid (``pair_grid`` in ``csrc/fock_lattice.h``): the rule
itself, and, with the oracle, that V_x psi, E_x and dE_x/domega on the working
grid equal those on the caller's grid for every kind of call that may take one
(cubic and general cells, both kernels, uneven occupations, trial orbitals, k
points), up to the oracle's own rounding: FP64 transforms of length N^3 differ by
about u log2(N^3) ~ 2e-15 of the largest value; the bound is 1e-12.  CPU only."""

import subprocess

import numpy as np
import pytest

import oracle
from paper_1305_7313_gb300 import synth
from tests._common import cubic, host_program, rel_inf

SIZES = sorted({8, 12, 16, 24, 32, 36, 48, 64, 72, 96} | {20, 28, 40, 56, 60, 80})
SKEW = np.array([[1.0, 0.04, 0.0], [0.03, 1.0, 0.02], [0.0, -0.03, 1.0]])


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    exe = host_program("pair_grid_driver.cpp", tmp_path_factory.mktemp("pair_grid"))
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    return {(int(a), int(b)): int(c) for a, b, c in (line.split() for line in out.splitlines())}


def test_the_rule_takes_the_smallest_grid_without_aliasing(rule):
    for (n, reach), s in rule.items():
        fits = [x for x in SIZES if 2 * reach < x < n]
        assert s == (fits[0] if fits else n), (n, reach)
        if 2 * reach >= n:
            assert s == n, (n, reach)  # an aliasing grid is its own operator


def reach_of(mill):
    return 2 * int(np.max(np.abs(mill)))


@pytest.mark.parametrize("n,cell,ecut,kind,omega,expect", [
    (24, cubic(6.4), 12.0, "spencer_alavi", None, 20),
    (32, cubic(8.5), 12.0, "erfc", 0.3, 28),
    (36, cubic(10.125), 12.0, "erfc", 0.106, 32),
    (32, (8.3 * SKEW).ravel(), 12.0, "erfc", 0.3, 28),
    (48, cubic(9.0), 8.0, "spencer_alavi", None, 24),
    (24, cubic(10.0), 10.0, "spencer_alavi", None, 24),  # aliases: kept
])
def test_the_operator_is_the_same_on_the_working_grid(rule, n, cell, ecut, kind, omega, expect):
    mill, _ = oracle.gsphere((n, n, n), cell, ecut)
    s = rule[n, reach_of(mill)]
    assert s == expect
    c = synth.orbitals(mill, cell, 4, 11)
    occ = np.array([2.0, 1.5, 0.7, -0.2])
    v, e, d = oracle.fock_apply(c, occ, mill, (n, n, n), cell, kind, omega)
    vs, es, ds = oracle.fock_apply(c, occ, mill, (s, s, s), cell, kind, omega)
    assert rel_inf(vs, v) <= 1e-12 and abs(es - e) <= 1e-12 * abs(e) and abs(ds - d) <= 1e-12 * max(abs(d), 1e-300)


@pytest.mark.parametrize("n,length,ecut,expect", [(24, 6.5, 8.0, 20), (32, 7.9, 12.0, 28), (36, 9.2, 12.0, 32)])
def test_k_points_are_the_same_on_the_working_grid(rule, n, length, ecut, expect):
    kpts = np.array([[0.0, 0.0, 0.0], [0.5, 0.0, 0.0], [0.25, -0.25, 0.5]])
    wk = np.array([0.5, 0.3, 0.2])
    cell = cubic(length)
    mills = [oracle.gsphere_k((n, n, n), cell, ecut, k)[0] for k in kpts]
    reach = max(int(np.max(b.max(0) - a.min(0))) for a in mills for b in mills)
    s = rule[n, reach]
    assert s == expect
    c = [synth.orbitals_k(m, cell, k, 2, 20 + i) for i, (m, k) in enumerate(zip(mills, kpts))]
    occ = np.array([[2.0, 1.0]] * 3)
    v, e = oracle.fock_apply_kpoints(c, occ, mills, kpts, wk, (n, n, n), cell, "erfc", 0.4)
    vs, es = oracle.fock_apply_kpoints(c, occ, mills, kpts, wk, (s, s, s), cell, "erfc", 0.4)
    assert abs(es - e) <= 1e-12 * abs(e)
    for a, b in zip(vs, v):
        assert rel_inf(a, b) <= 1e-12
