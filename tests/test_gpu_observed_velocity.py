"""The velocity behind spectra, band energies and column means is v = u / u^0 of the fields that
rlbm_moments hands out: FP32 and 16-bit states to two-float precision.  v is formed to 2^-44, the sums
and transforms (fewer than a hundred two-float operations of 2^-46) keep it to 2^-39: 2^-38 of the largest
value."""
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


@pytest.mark.parametrize("precision", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("flow", [0.0, 0.02, 0.1, 0.7])
@pytest.mark.parametrize("nx,ny,masked", [(64, 48, False), (96, 63, True)])
def test_observations_use_the_fields_velocity(R, precision, flow, nx, ny, masked):
    e, ux, uy = inputs.smooth_random_fields(nx, ny, seed=4, eps_amp=1e-3, u_amp=2e-3, kmax=3)
    solid = np.zeros((ny, nx), np.uint8)
    if masked:
        solid[10:21, 30:44] = 1
    lat = R.Lattice(nx, ny, precision=precision, eta_over_s=0.1, solid=solid if masked else None, init_eps=e, init_ux=ux + flow,
                    init_uy=uy - 0.5 * flow)
    lat.step(4)
    _, U, V, _ = lat.moments()
    u0 = np.sqrt(1.0 + U * U + V * V)
    vx, vy = U / u0, V / u0
    jx, jy = lat.column_means()
    vmax = max(np.abs(vx).max(), np.abs(vy).max())
    assert np.abs(jx - vx.mean(0)).max() <= 2.0 ** -38 * vmax and np.abs(jy - vy.mean(0)).max() <= 2.0 ** -38 * vmax
    P = 0.5 * (np.abs(np.fft.fft2(vx)) ** 2 + np.abs(np.fft.fft2(vy)) ** 2) / (nx * ny) ** 2
    kx, ky = (np.rint(np.fft.fftfreq(n) * n).astype(np.int64) for n in (nx, ny))
    k2 = ky[:, None] ** 2 + kx[None, :] ** 2
    n = np.rint(np.sqrt(k2)).astype(np.int64)
    ref = np.bincount(n.ravel(), P.ravel())
    assert np.abs(lat.spectrum(ref.size) - ref).max() <= 2.0 ** -38 * ref.max()
    assert abs(lat.band_energy(0, 0) - P.sum()) <= 2.0 ** -38 * P.sum()
    lat.close()
