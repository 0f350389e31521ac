"""Spectra and band energies of FP32 states whose velocities lie far below 1: FP32 deviations reach down
to 1e-38, and the squares of such velocities below FP32's range still count.  Against numpy on the
fields of the same state, 2^-20 of the largest bin, the bar of FP32 states at ordinary velocities."""
import os

import numpy as np
import pytest

from paper_2205_04658_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_04658_gb300 import build as B
    from paper_2205_04658_gb300 import rlbm
    if not os.path.exists(rlbm.LIB_PATH):
        B.build()
    return rlbm


# (columns in shared memory, and rows and columns too long for it)
@pytest.mark.parametrize("nx,ny", [(64, 48), (24, 6600), (6600, 8)])
@pytest.mark.parametrize("precision", ["f32", "bf16"])
@pytest.mark.parametrize("amp", [1e-2, 1e-14, 1e-20, 1e-24, 1e-30])
def test_spectrum_of_small_velocities(R, precision, amp, nx, ny):
    _, ux, uy = inputs.smooth_random_fields(nx, ny, seed=5, u_amp=1.0, kmax=3)
    lat = R.Lattice(nx, ny, precision=precision, init_ux=amp * ux, init_uy=amp * uy)
    E, UX, UY, _ = lat.moments()
    u0 = np.sqrt(1.0 + UX * UX + UY * UY)
    P = 0.5 * (np.abs(np.fft.fft2(UX / u0)) ** 2 + np.abs(np.fft.fft2(UY / u0)) ** 2) / (nx * ny) ** 2
    kx, ky = (np.rint(np.fft.fftfreq(n) * n).astype(np.int64) for n in (nx, ny))
    k2 = ky[:, None] ** 2 + kx[None, :] ** 2
    n = np.rint(np.sqrt(k2)).astype(np.int64)
    ref = np.bincount(n.ravel(), P.ravel())
    assert ref.max() > 0.01 * amp * amp  # the state holds the velocities it was given
    assert np.abs(lat.spectrum(ref.size) - ref).max() <= 2.0 ** -20 * ref.max()
    assert abs(lat.band_energy(1, 9) - P[(k2 >= 1) & (k2 < 9)].sum()) <= 2.0 ** -20 * P.sum()
    lat.close()
