"""The double-float FP64 stage with more than 1024 projectors, whose h c then
comes from global memory, against the plain FP64 stage: 1125 projectors (125
atoms, l <= 2) and 1331 (one each).

Tolerance: H u as against the oracle, 1e-12 of the largest value (48-bit
products against 53-bit ones: ~4e-15 of the largest term, the kinetic diagonal's
~1e2 times u); three steps as in the split stage's test, 2e-13 and a factor five.
"""
import dataclasses

import numpy as np
import pytest

from paper_0812_2801_gb300 import emd, inputs

pytestmark = pytest.mark.gpu


def _system(n, h, cells, species):
    R = inputs.jitter(inputs.lattice_sites("sc", cells, n * h / cells), seed=3, amp=0.05)
    s = inputs.small_system(n=n, h=h, fd_order=8, n_atoms=2, seed=5, n_orb=3)
    return dataclasses.replace(s, R=np.ascontiguousarray(R), V=np.zeros_like(R), species=species)


@pytest.mark.parametrize("n,h,cells,lmax", [(24, 0.5, 5, 2), (44, 0.5, 11, 0)])
def test_matches_plain_fp64_stage(n, h, cells, lmax):
    sp = dataclasses.replace(inputs.SI_LIKE, r_c=0.4, r_proj=1.1 if lmax else 0.9, a_loc=0.4,
                             r_loc=1.1, lmax=lmax, h_l=(0.6, -0.35))
    s = _system(n, h, cells, sp)
    assert s.n_atoms * (lmax + 1) ** 2 > 1024
    rng = np.random.default_rng(7)
    u = rng.normal(size=(3, n, n, n)) + 1j * rng.normal(size=(3, n, n, n))
    got = []
    for variant in (1, 0):
        g = emd.System(s)
        emd.emd_set_option(g.handle, emd.EMD_OPT_STAGE_VARIANT, variant)
        Hu = emd.emd_apply_hamiltonian(g.handle, u)
        g.propagate(3, dt=0.005, mu=1.0)
        got.append((Hu, g.state()[2], g.state()[3]))
        g.close()
    for a, b in zip(*got):
        assert np.isfinite(a).all()
        assert np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(a))
    assert not np.array_equal(got[0][0], got[1][0])     # two different stages ran
