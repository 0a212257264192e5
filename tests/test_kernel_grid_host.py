"""The Gamma-point kernel tables (``grid_kernel`` in ``csrc/fock_lattice.h``): the
mean of v(k) and v(-k), which is the operator of the sum over the full grid for real
pair densities.  Against the oracle's kernels on the full grid to 1e-13 of their
largest value (the same FP64 expressions, a few roundings apart), and, with random
real densities, against its potential and energies; both bounds also hold where the
two values differ, on the Nyquist planes of the hexagonal cell.  CPU only."""

import subprocess

import numpy as np
import pytest

from oracle.fock import kernel_grid, pair_energy, pair_potential
from tests._common import host_program, rel_inf

CELLS = [5.0 * np.eye(3), np.array([[5.0, 0.0, 0.0], [-2.5, 2.5 * np.sqrt(3.0), 0.0], [0.0, 0.0, 5.0]])]
KINDS = ["spencer_alavi", "erfc"]


@pytest.fixture(scope="module")
def tables(tmp_path_factory):
    exe = host_program("kernel_grid_driver.cpp", tmp_path_factory.mktemp("kernel_grid"))
    out = {}
    for line in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines():
        w = line.split()
        c, kind, n, k1, k2, k3 = (int(x) for x in w[:6])
        t = out.setdefault((c, kind, n), np.zeros((2, n, n, n // 2 + 1)))
        t[:, k1, k2, k3] = [float.fromhex(x) for x in w[6:]]
    return out


def negated(v):
    """v at -k (indices modulo n)."""
    return np.roll(v[::-1, ::-1, ::-1], 1, axis=(0, 1, 2))


@pytest.mark.parametrize("n", [8, 7])
@pytest.mark.parametrize("kind", [0, 1], ids=KINDS)
@pytest.mark.parametrize("cell", [0, 1], ids=["cubic", "hexagonal"])
def test_the_table_is_the_operator_of_the_full_grid(tables, cell, kind, n):
    table = tables[cell, kind, n]
    full = kernel_grid(KINDS[kind], (n,) * 3, CELLS[cell], 0.3)
    for t, f in zip(table, full):
        scale = max(np.abs(f).max(), 1e-300)
        assert np.abs(t - 0.5 * (f + negated(f))[:, :, : n // 2 + 1]).max() <= 1e-13 * scale
    v, _ = full
    differ = np.abs(v - negated(v)).max() > 1e-3 * v.max()
    assert differ == (cell == 1 and n % 2 == 0)
    # through the half spectrum, as the passes use it
    rng = np.random.default_rng(n)
    a, b = rng.standard_normal((2, n, n, n))
    half = np.fft.rfftn(a * b)
    phi = np.fft.irfftn(table[0] * half, s=(n,) * 3, axes=(0, 1, 2))
    assert rel_inf(phi, pair_potential(a, b, v).real) <= 1e-13
    weight = np.full(n // 2 + 1, 2.0)
    weight[0] = 1.0
    if n % 2 == 0:
        weight[-1] = 1.0
    e = np.sum(weight * table[0] * np.abs(half) ** 2) / n ** 6
    assert abs(e - pair_energy(a, b, v)) <= 1e-13 * e
