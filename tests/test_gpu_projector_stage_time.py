"""The double-float stage's time with nine projectors per atom at order 8,
against order 6 on the same 96^3 grid (32 orbitals).

Bound: the ratio of the two orders' stencil operations, (78 + 56 4) / (78 + 56
3) = 1.23.  The projector term, most of the time here, is the same in both, so a
kernel whose record loads are as well overlapped at order 8 stays below it.
"""
import dataclasses

import numpy as np
import pytest

from paper_0812_2801_gb300 import emd, inputs

pytestmark = pytest.mark.gpu


def _stage_ms(s):
    g = emd.System(s, emd.EMD_FP64)
    g.propagate(1)
    emd.emd_set_option(g.handle, emd.EMD_OPT_PROFILE, 1)
    g.propagate(3)
    g.forces()
    ms, n = emd.emd_kernel_stats(g.handle)
    g.close()
    return ms / n


def test_order_8_costs_no_more_than_its_operations():
    b = inputs.precision_c96(10.0)
    sp = dataclasses.replace(b.species, lmax=2, h_l=(0.6, -0.35))
    s = dataclasses.replace(b, psi=np.ascontiguousarray(b.psi[:32]), species=sp)
    o8 = _stage_ms(s)
    o6 = _stage_ms(dataclasses.replace(s, fd_order=6))
    assert o8 <= 302.0 / 246.0 * o6, (o8, o6)
