"""The structure factor's DFT passes at the sizes where their kernels change:
shared rows and one row per thread, the general x pass (more than 18 kept k_x), one
and four wavevector pairs per block, planar fields (which end with the y pass), odd and
even axes (with and without a self-conjugate k) and windows."""
import numpy as np
import pytest

import paper_1104_0078_gb300 as F

pytestmark = pytest.mark.gpu


def _axis(n, kmax):
    return np.arange(n) if kmax <= 0 or 2 * kmax + 1 >= n else np.r_[0:kmax + 1, n - kmax:n]


@pytest.mark.parametrize("nx,ny,nz,kmax", [(64, 64, 64, 0), (64, 64, 1, 0), (300, 20, 1, 16), (2048, 12, 1, 17),
                                           (130, 4, 4, 0), (7, 5, 9, 0), (40, 33, 96, 7), (256, 256, 300, 1),
                                           (35, 36, 37, 17), (8, 700, 4, 3)])
def test_spectrum_against_numpy(nx, ny, nz, kmax):
    dim = 2 if nz == 1 else 3
    p = F.flb_params_default(dim=dim, q=9 if dim == 2 else 19, nx=nx, ny=ny, nz=nz, sq_kmax=kmax)
    psi = np.random.default_rng(nx + ny + nz).standard_normal((nz, ny, nx)).astype(np.float32).astype(np.float64)
    s = F.Solver(p)
    s.set_fields(psi=psi)
    s.sample(1)
    s.sample(1)  # accumulates: the mean of two equal samples
    got, n = s.structure_factor()
    assert n == 2
    ref = np.abs(np.fft.fftn(psi)) ** 2 / psi.size
    ref = ref[np.ix_(_axis(nz, kmax), _axis(ny, kmax), _axis(nx, kmax))].reshape(-1)
    # binary32 sums of at most 256 terms in a chain along x and y: a component is off by
    # less than 256 * 2^-24 = 1.6e-5 of its rms, a square by twice its modulus times that
    assert np.all(np.abs(got - ref) <= 4e-5 * (ref + ref.mean()))
