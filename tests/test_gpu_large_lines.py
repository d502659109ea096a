"""Spectral solves whose lines take more than 48 KB of shared memory (grids
above about 170 points), even and odd, against numpy's FFT in FP64.

Tolerance as for the smaller grids: an FP64 FFT of N points is off by ~eps
log2(N) of the norm, ~2e-15 forward and back; 1e-13 of the largest value leaves
more than a factor ten.
"""
import numpy as np
import pytest

from oracle import emd_oracle as O
from paper_0812_2801_gb300 import emd, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [176, 189, 192])
def test_hartree_potential(n):
    s = inputs.small_system(n=n, h=0.3, fd_order=2, n_atoms=1, seed=n, n_orb=1)
    g = emd.System(s)
    _, _, _, rho = g.state(want_psi=False)
    v = emd.emd_get_potentials(g.handle, n)
    g.close()
    for got, q in ((v["v_h"], rho), (v["v_loc"], -v["g_ion"])):
        ref = O.poisson(q, s.h)
        assert np.max(np.abs(got - ref)) <= 1e-13 * np.max(np.abs(ref))
