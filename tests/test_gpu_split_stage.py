"""The double-float stage on split sets (csrc/stage_df.cu): 16 x 8 tiles that
overhang the grid, z-chunks of one plane up to the whole column, every order,
and the split copy of psi that one MD step leaves for the next.

Tolerance against the plain FP64 stage: a stage adds at most a few 2^-48 times
tau lambda_max / k <= 3 of the largest value, about 3e-14 per exponential, so
2e-13 over the three steps here; 1e-12 leaves a factor five.
"""
import numpy as np
import pytest

from paper_0812_2801_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def emd():
    from paper_0812_2801_gb300 import emd as E
    E.load()
    return E


def _run(emd, s, options, steps=3):
    g = emd.System(s)
    for k, v in options:
        emd.emd_set_option(g.handle, k, v)
    g.propagate(steps, dt=0.02, mu=1.0)
    out = g.state()
    g.close()
    return out


@pytest.mark.parametrize("n,order,atoms,n_orb", [
    (16, 8, 2, 3), (18, 6, 2, 4), (21, 8, 3, 5), (25, 4, 2, 1), (33, 2, 3, 6), (35, 8, 2, 4)])
def test_split_sets_match_plain_fp64(emd, n, order, atoms, n_orb):
    s = inputs.small_system(n=n, h=0.4, fd_order=order, n_atoms=atoms, seed=n, n_orb=n_orb)
    ref = _run(emd, s, [(emd.EMD_OPT_STAGE_VARIANT, 1)])
    first = None
    for zc in (0, 1, 5, n):
        got = _run(emd, s, [(emd.EMD_OPT_ZCHUNK, zc)])
        assert np.max(np.abs(got[2] - ref[2])) <= 1e-12 * np.max(np.abs(ref[2]))
        assert np.max(np.abs(got[3] - ref[3])) <= 1e-12 * np.max(np.abs(ref[3]))
        if first is None:
            first = got
        assert np.array_equal(got[2], first[2]) and np.array_equal(got[0], first[0])


def test_split_copy_is_dropped_when_it_goes_stale(emd):
    """H applications overwrite the set that holds psi's split values, and the
    plain stage and the point-major projections leave none: the trajectory's
    bits do not depend on what came between the steps."""
    s = inputs.small_system(n=20, h=0.35, fd_order=4, n_atoms=2, seed=3)
    a, b = emd.System(s), emd.System(s)
    a.propagate(9, dt=0.02, mu=1.0)
    for _ in range(9):
        b.propagate(1, dt=0.02, mu=1.0)
        emd.emd_apply_hamiltonian(b.handle, s.psi)
        assert emd.emd_get_projections(b.handle, s.n_atoms, s.n_orb).shape == (2, s.n_orb)
    for x, y in zip(a.state(), b.state()):
        assert np.array_equal(x, y)
    # switching to the plain stage and back, the same on both (one in single steps)
    for g, cut in ((a, [4]), (b, [1, 1, 1, 1])):
        emd.emd_set_option(g.handle, emd.EMD_OPT_STAGE_VARIANT, 1)
        g.propagate(2, dt=0.02, mu=1.0)
        emd.emd_set_option(g.handle, emd.EMD_OPT_STAGE_VARIANT, 0)
        for k in cut:
            g.propagate(k, dt=0.02, mu=1.0)
    for x, y in zip(a.state(), b.state()):
        assert np.array_equal(x, y)
    # new orbitals restart from them
    psi = a.state()[2]
    emd.emd_set_orbitals(b.handle, psi)
    emd.emd_set_orbitals(a.handle, psi)
    a.propagate(2, dt=0.02, mu=1.0)
    b.propagate(2, dt=0.02, mu=1.0)
    assert np.array_equal(a.state()[2], b.state()[2])
    a.close()
    b.close()
