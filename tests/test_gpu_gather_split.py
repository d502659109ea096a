"""The atom-major double-float gathers when one CTA, or 2, 4 or 8 CTAs, share
an atom's entries (csrc/emd_internal.cuh, emd_gather_split): projections
against the oracle, and the same bits on a second call for projections and
forces.

Tolerance: a projection sums up to ~1e4 terms of 48-bit values, so 2^-48 per
term with random signs stays below 1e-13 of the largest projection; 1e-12
leaves a factor ten.
"""
import dataclasses

import numpy as np
import pytest

from oracle import emd_oracle as O
from paper_0812_2801_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def emd():
    from paper_0812_2801_gb300 import emd as E
    E.load()
    return E


# (n, h, r_proj, atoms, lmax): the table capacity (2 ceil(r / h) + 3)^3, or 8
# n^3 if smaller, over 2048 bounds the split, and so do atoms x blocks
@pytest.mark.parametrize("n,h,r_proj,atoms,lmax", [
    (20, 0.5, 3.0, 3, 0),     # capacity 3375: one CTA
    (20, 0.5, 4.4, 3, 0),     # 9261: two
    (24, 0.4, 4.6, 2, 0),     # 19683: eight allowed by the pairs, four by the capacity
    (24, 0.4, 4.79, 1, 2),    # eight, nine projectors
    (21, 0.35, 7.0, 1, 0),    # spheres that wrap the box: several images per point
    (18, 0.4, 5.0, 7, 1),     # 196 pairs
])
def test_split_gathers_match_oracle(emd, n, h, r_proj, atoms, lmax):
    sp = dataclasses.replace(inputs.SI_LIKE, r_proj=r_proj, r_loc=3.0, lmax=lmax, h_l=(0.6, 0.4))
    s = inputs.small_system(n=n, h=h, fd_order=4, n_atoms=atoms, seed=5, species=sp)
    st = O.init_state(s)
    ref = O.projections(st.psi, st.tables, sp, h)
    g = emd.System(s)
    nch = (lmax + 1) ** 2
    c = emd.emd_get_projections(g.handle, s.n_atoms, s.n_orb, nch)
    F = g.forces()
    assert np.max(np.abs(c - ref)) <= 1e-12 * np.max(np.abs(ref))
    emd.emd_set_ions(g.handle, s.R, s.V)          # recompute everything
    assert np.array_equal(emd.emd_get_projections(g.handle, s.n_atoms, s.n_orb, nch), c)
    assert np.array_equal(g.forces(), F)
    g.close()
