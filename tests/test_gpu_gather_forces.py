"""Forces of the atom-major double-float gathers against the oracle, for 1, 2, 4
and 8 CTAs per (projector, orbital block), limited by the table's capacity or
by the number of pairs.

Tolerance, per atom: a projection c and its derivative dc are sums of products
of 48-bit values (about three roundings of 2^-48 of each term's magnitude), so
the nonlocal force is off by at most 3 2^-48 sum 2 occ |h| (C |dc| + |c| D) with
C and D the sums of magnitudes; the density carries the same relative error
into the potential that the local force multiplies, so that is off by at most
3 2^-48 (2 / a^2) h^3 max|v| sum |g d|.  Both are 2e-14 of these magnitudes with
the oracle's own rounding; 1e-13 leaves a factor five.  The short-range ion
force is plain FP64.  (A bound relative to the force itself does not hold: it is
what is left of these magnitudes, 1e-7 of 30 for a single atom.)
"""
import dataclasses

import numpy as np
import pytest

from oracle import emd_oracle as O
from paper_0812_2801_gb300 import emd, inputs

pytestmark = pytest.mark.gpu


def _split(n, h, r_proj, pairs):
    """The launch rule (csrc/launch_rules.h) and the capacity it is given."""
    cube = (2 * int(np.ceil(r_proj / h)) + 3) ** 3
    cap = min(n ** 3, cube) if n * h > 2 * r_proj else min(8 * n ** 3, 27 * cube)
    s = 1
    while s < 8 and pairs * s < 152 * 12 and cap // 2 >= 2048 * s:
        s *= 2
    return s


def _magnitudes(st):
    sp, h3 = st.sp, st.h ** 3
    v = np.max(np.abs(st.v_h + st.v_loc))
    flat = st.psi.reshape(st.psi.shape[0], -1)
    c = O.projections(st.psi, st.tables, sp, st.h)
    ch = O.channels(sp)
    out = np.zeros(st.R.shape[0])
    for j, (_, dx, dy, dz) in enumerate(st.tables.loc):
        g = O.gaussian_charge_values(sp, dx, dy, dz)
        out[j] += 2.0 / sp.a_loc ** 2 * h3 * v * max(np.sum(np.abs(g * d)) for d in (dx, dy, dz))
    for j, (idx, dx, dy, dz) in enumerate(st.tables.proj):
        u = np.abs(flat[:, idx])
        for k, (l, m) in enumerate(ch):
            P = j * len(ch) + k
            C = h3 * (u @ np.abs(O.projector_lm_values(sp, l, m, dx, dy, dz)))
            for g in O.projector_lm_gradient(sp, l, m, dx, dy, dz):
                dc = np.abs(flat[:, idx] @ g) * h3
                D = h3 * (u @ np.abs(g))
                out[j] += 2.0 * abs(st.tables.hP[P]) * st.occ * np.sum(C * dc + np.abs(c[P]) * D)
    _, sr = O.short_range_ion(st.R, sp, st.psi.shape[1] * st.h)
    return out + np.max(np.abs(sr))


@pytest.mark.parametrize("n,h,r_proj,atoms,lmax,split", [
    (20, 0.5, 3.0, 3, 0, 1),     # capacity 3375
    (20, 0.5, 4.4, 3, 0, 2),     # 8000
    (24, 0.4, 4.6, 2, 0, 4),     # 13824
    (26, 0.38, 4.9, 2, 2, 8),    # 17576, nine projectors
    (21, 0.35, 7.0, 2, 0, 8),    # spheres that wrap the box: several images per point
    (26, 0.38, 4.9, 8, 2, 4),    # 17576, but 576 pairs
    (18, 0.4, 5.0, 7, 1, 8),     # 46656, 196 pairs, several channels
])
def test_forces_match_oracle(n, h, r_proj, atoms, lmax, split):
    sp = dataclasses.replace(inputs.SI_LIKE, r_proj=r_proj, r_loc=3.0, lmax=lmax, h_l=(0.6, 0.4))
    s = inputs.small_system(n=n, h=h, fd_order=4, n_atoms=atoms, seed=5, species=sp)
    assert _split(n, h, r_proj, atoms * (lmax + 1) ** 2 * ((s.n_orb + 1) // 2)) == split
    st = O.init_state(s)
    g = emd.System(s)
    off = np.max(np.abs(g.forces() - st.F), axis=1)
    g.close()
    assert np.all(off <= 1e-13 * _magnitudes(st)), off / _magnitudes(st)
