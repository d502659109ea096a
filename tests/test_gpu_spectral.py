"""The five-kernel spectral solve (csrc/fft2.cu) against numpy's FFT in FP64:
every butterfly of 2 to 16 points, two to four factors, even and odd
grids, an 8-byte aligned grid, and the
solve in place.

Tolerance: an FP64 FFT of N points is off by ~eps log2(N) of the norm, ~2e-15
forward and back; 1e-13 of the largest value leaves more than a factor ten.
"""
import numpy as np
import pytest

from oracle import emd_oracle as O
from paper_0812_2801_gb300 import emd, inputs

pytestmark = pytest.mark.gpu

# n and (even n) n / 2 cover every butterfly and two to four factors
SIZES = [2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16, 18, 20, 21, 22, 24, 25, 26, 27, 28, 30, 32, 33,
         35, 36, 39, 40, 42, 44, 45, 48, 49, 50, 52, 54, 55, 56, 60, 63, 64]


def _ref(q, h):
    return O.poisson(q, h)


@pytest.mark.parametrize("n", SIZES)
def test_poisson_static_sizes(n):
    import torch
    q = np.random.default_rng(n).normal(size=(n, n, n))
    ref = _ref(q, 0.3)
    # one extra value in front: 8-byte, not 16-byte aligned
    buf = torch.zeros(n ** 3 + 1, dtype=torch.float64, device="cuda")
    buf[1:] = torch.from_numpy(q.ravel()).cuda()
    out = torch.full((n ** 3 + 1,), float("nan"), dtype=torch.float64, device="cuda")
    emd.emd_poisson_static(n, 0.3, buf.data_ptr() + 8, out.data_ptr() + 8)
    got = out[1:].cpu().numpy().reshape(n, n, n)
    assert np.isnan(out[0].item())
    assert np.max(np.abs(got - ref)) <= 1e-13 * np.max(np.abs(ref))
    emd.emd_poisson_static(n, 0.3, buf.data_ptr() + 8, buf.data_ptr() + 8)   # in place
    assert np.array_equal(buf[1:].cpu().numpy().reshape(n, n, n), got)


@pytest.mark.parametrize("n", [65, 66, 77, 78, 91, 98, 99, 104, 110, 117, 121, 125, 143])
def test_hartree_potential_sizes(n):
    """Larger grids through the library's own solve (no ions: rho of one orbital)."""
    s = inputs.small_system(n=n, h=0.3, fd_order=2, n_atoms=1, seed=n, n_orb=1)
    g = emd.System(s)
    _, _, _, rho = g.state(want_psi=False)
    v = emd.emd_get_potentials(g.handle, n)
    g.close()
    for got, q in ((v["v_h"], rho), (v["v_loc"], -v["g_ion"])):
        ref = _ref(q, 0.3)
        assert np.max(np.abs(got - ref)) <= 1e-13 * np.max(np.abs(ref))
