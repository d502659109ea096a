"""The double-float stage's time as the projectors pass 1024, from where their
h c comes from global memory: 10^3 and 11^3 atoms on the same 64^3 grid, order 8,
16 orbitals.

Bound: 1.331, the ratio of the projector entries per point, as if the entries
were all of the stage.  (They are a small part here, so the rest of the stage
must not change its form at the limit.)
"""
import dataclasses

import numpy as np
import pytest

from paper_0812_2801_gb300 import emd, inputs

pytestmark = pytest.mark.gpu


def _stage_ms(cells):
    n, h = 64, 0.375
    rng = np.random.default_rng(1)
    R = inputs.jitter(inputs.lattice_sites("sc", cells, n * h / cells), seed=3, amp=0.05)
    psi = rng.normal(size=(16, n, n, n)) + 1j * rng.normal(size=(16, n, n, n))
    psi /= np.sqrt(h ** 3 * np.sum(np.abs(psi) ** 2, axis=(1, 2, 3), keepdims=True))
    sp = dataclasses.replace(inputs.SI_LIKE, r_c=0.6, r_proj=2.0, a_loc=0.5, r_loc=2.0)
    s = inputs.small_system(n=16, h=h, fd_order=8, n_atoms=2, seed=5)
    g = emd.System(dataclasses.replace(s, n=n, R=np.ascontiguousarray(R), V=np.zeros_like(R),
                                       psi=psi, species=sp))
    g.propagate(1, dt=0.002, mu=1.0)
    emd.emd_set_option(g.handle, emd.EMD_OPT_PROFILE, 1)
    g.propagate(3, dt=0.002, mu=1.0)
    g.forces()
    ms, k = emd.emd_kernel_stats(g.handle)
    g.close()
    return ms / k


def test_no_step_in_the_time_at_1024_projectors():
    few, many = _stage_ms(10), _stage_ms(11)
    assert many <= 1.331 * few, (few, many)
