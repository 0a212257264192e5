"""General cells whose grid aliases the pair densities (N <= 2 reach): there the
spectra reach the Nyquist planes, where G and -G differ in length, against the
oracle's sum over the full grid with the tolerances of the parity tests."""

import numpy as np
import pytest

import oracle
from oracle.fock import kernel_grid
from paper_1305_7313_gb300 import FockPlan, _lib, synth
from tests._common import rel_inf, require_gpu

pytestmark = pytest.mark.gpu

TOL = {_lib.PREC_FP64: (1e-10, 1e-10), _lib.PREC_DF64: (1e-10, 1e-10), _lib.PREC_MIXED32: (2e-5, 5e-6)}
SHAPES = {
    "hexagonal": np.array([[1.0, 0.0, 0.0], [-0.5, np.sqrt(0.75), 0.0], [0.0, 0.0, 1.0]]),
    "monoclinic": np.array([[1.0, 0.0, 0.0], [0.0, 1.0, 0.0], [0.25, 0.0, 1.0]]),
    "triclinic": np.array([[1.0, 0.1, 0.0], [-0.2, 1.0, 0.15], [0.05, -0.1, 1.0]]),
}
CASES = [(8, 4.2, 6.0, "hexagonal", _lib.SPENCER_ALAVI), (24, 10.0, 10.0, "hexagonal", _lib.ERFC),
         (24, 10.0, 10.0, "triclinic", _lib.SPENCER_ALAVI), (32, 13.5, 10.0, "monoclinic", _lib.ERFC)]


@pytest.mark.parametrize("prec", sorted(TOL), ids=["fp64", "mixed32", "df64"])
@pytest.mark.parametrize("n,length,ecut,shape,kernel", CASES, ids=["%d-%s" % (c[0], c[3]) for c in CASES])
def test_aliasing_grids_of_general_cells(n, length, ecut, shape, kernel, prec):
    torch = require_gpu()
    cell = length * SHAPES[shape]
    mill, _ = oracle.gsphere((n,) * 3, cell, ecut)
    assert n <= 4 * np.abs(mill).max()  # it aliases
    c = synth.orbitals(mill, cell, 4, n)
    occ = np.array([2.0, 1.5, 1.0, 0.5])
    omega = 0.3 if kernel == _lib.ERFC else None
    name = "erfc" if kernel == _lib.ERFC else "spencer_alavi"
    tv, te = TOL[prec]
    with FockPlan(n, cell, ecut, kernel, omega, prec) as plan:
        psi = torch.from_numpy(c).cuda()
        v, e, d = plan.apply(psi, occ, want_dex=True)
        pairs = [(0, 0), (0, 3), (2, 1)]
        pe, _ = plan.pair_energies(psi, pairs, want_d=True)
        plan.set_occupied(psi[:2].contiguous(), occ[:2])
        fixed = plan.apply_fixed(psi[2:].contiguous())
    vr, er, dr = oracle.fock_apply(c, occ, mill, (n,) * 3, cell, name, omega)
    assert rel_inf(v.cpu().numpy(), vr) <= tv
    assert abs(e - er) <= te * abs(er) and abs(d - dr) <= te * abs(dr)
    fr = oracle.fock_apply_to(c[:2], occ[:2], c[2:], mill, (n,) * 3, cell, name, omega)
    assert rel_inf(fixed.cpu().numpy(), fr) <= tv
    vg, dvg = kernel_grid(name, (n,) * 3, cell, omega)
    real = oracle.orbitals_to_real(c, mill, (n,) * 3, cell, real=True)
    for k, (i, j) in enumerate(pairs):
        ref = oracle.pair_energy(real[i], real[j], vg, dvg)[0]
        assert abs(pe[k] - ref) <= te * abs(ref)
