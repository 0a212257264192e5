"""The DFTs of radix 5, 7, 10, 14, 15, 18, 20 and 24 (``Dft`` in
``csrc/fft_core.cuh``), compiled for the host, against the DFT evaluated in FP64
on the same inputs.  Bound: at most six levels of sums (8 x 3 and its inner
constants, a twiddle product), each within 4 u of the sum of the inputs' moduli:
24 u.  CPU only."""

import subprocess

import numpy as np
import pytest

from tests._common import host_program

RADICES = (5, 7, 10, 14, 15, 18, 20, 24)


@pytest.fixture(scope="module")
def cases(tmp_path_factory):
    exe = host_program("dft_composites_driver.cu", tmp_path_factory.mktemp("dft"))
    got = {}
    for line in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines():
        f = line.split()
        v = np.array([float(t) for t in f[4:]])
        got[tuple(int(t) for t in f[:4])] = (v[0::2] + 1j * v[1::2]).reshape(3, int(f[1]))
    return got


@pytest.mark.parametrize("radix", RADICES)
@pytest.mark.parametrize("typ,u", [(0, 2.0**-24), (1, 2.0**-53)], ids=["float", "double"])
def test_composite_radices_match_the_direct_dft(cases, radix, typ, u):
    k = np.arange(radix)
    for sign in (-1, 1):
        for mode in (0, 1):
            x, w, y = cases[typ, radix, sign, mode]
            if mode == 1:
                x = np.concatenate([x[:1], x[1:] * w[1:]])
            ref = np.exp(sign * 2j * np.pi * (np.outer(k, k) % radix) / radix) @ x
            assert np.max(np.abs(y - ref)) <= 24 * u * np.sum(np.abs(x)), (sign, mode)
            assert np.max(np.abs(y - np.conj(np.exp(sign * 2j * np.pi * np.outer(k, k) / radix)) @ x)) > 1e-3
