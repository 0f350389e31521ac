"""Observations against numpy on the fields of the same state: the spectrum and band energies
(every route of the transform), the column means and the totals, at the edges of the kernels'
tiles and strips.  FP64 states: the transform's rounding is a few 1e-16 per stage (and per term
of a direct sum), so sums of its squares agree to 1e-12 of the largest; FP32 states carry FP32
fields (a few 2^-24 each, a mean over cells and a band's energy at most that, relative to the
largest)."""
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


def _velocity(E, UX, UY):
    u0 = np.sqrt(1.0 + UX * UX + UY * UY)
    return UX / u0, UY / u0


# strips of two and of four columns, a last strip that is not whole, rows and columns too long
# for shared memory (6600, 3400), radices 3, 5, 7 and prime factors above 8
@pytest.mark.parametrize("nx,ny", [(8, 8), (9, 13), (33, 47), (64, 105), (611, 22), (24, 3400), (6600, 8), (8, 6600)])
@pytest.mark.parametrize("precision,tol", [("f64", 1e-12), ("f32", 2.0 ** -20)])
def test_transforms_match_numpy(R, nx, ny, precision, tol):
    e, ux, uy = inputs.smooth_random_fields(nx, ny, seed=nx + ny, u_amp=0.05, kmax=3)
    lat = R.Lattice(nx, ny, precision=precision, init_eps=e, init_ux=ux, init_uy=uy)
    vx, vy = _velocity(*lat.moments()[:3])
    P = 0.5 * (np.abs(np.fft.fft2(vx)) ** 2 + np.abs(np.fft.fft2(vy)) ** 2) / (nx * ny) ** 2
    kx, ky = (np.rint(np.fft.fftfreq(n) * n).astype(np.int64) for n in (nx, ny))
    k2 = ky[:, None] ** 2 + kx[None, :] ** 2
    n = np.rint(np.sqrt(k2)).astype(np.int64)
    nbins = int(n.max()) + 3
    ref = np.bincount(n.ravel(), P.ravel(), nbins)
    assert np.abs(lat.spectrum(nbins) - ref).max() <= tol * ref.max()
    for lo, hi in ((0, 0), (0, 5), (5, 0), (2, 17)):
        want = P[(k2 >= lo) & ((k2 < hi) if hi else True)].sum()
        assert abs(lat.band_energy(lo, hi) - want) <= tol * P.sum()
    lat.close()


@pytest.mark.parametrize("precision,tol", [("f64", 1e-13), ("f32", 2.0 ** -22), ("f16", 2.0 ** -22)])
@pytest.mark.parametrize("nx,ny,walls", [(8, 8, 0), (33, 17, 0), (96, 50, 1), (31, 200, 1), (1200, 500, 0)])
def test_means_and_totals_match_the_fields(R, nx, ny, walls, precision, tol):
    e, ux, uy = inputs.smooth_random_fields(nx, ny, seed=7, eps_amp=0.02, u_amp=0.05, kmax=3)
    solid = np.zeros((ny, nx), np.uint8)
    if walls:
        solid[3:9, 5:12] = 1
    lat = R.Lattice(nx, ny, precision=precision, walls_y=walls, solid=solid if walls else None, eps0=1.25,
                    init_eps=1.25 * e, init_ux=ux, init_uy=uy)
    E, UX, UY, tot = lat.moments()
    jx, jy = lat.column_means()
    assert np.array_equal(lat.totals(), tot)
    lat.close()
    fluid = solid == 0
    assert np.all(E[~fluid] == 0.0) and np.all(UX[~fluid] == 0.0) and np.all(E[fluid] > 0.0)
    vx, vy = _velocity(E, UX, UY)
    assert np.abs(jx - vx.mean(0)).max() <= tol * 0.05 and np.abs(jy - vy.mean(0)).max() <= tol * 0.05
    assert abs(tot[3] - 0.5 * (vx * vx + vy * vy).sum()) <= 4 * tol * tot[3]
    # T^00 = (4/3 eps u^0 u^0 - eps/3) of the ideal part; the start is an equilibrium pulled once
    ideal = (E * (4.0 * (1.0 + UX * UX + UY * UY) - 1.0) / 3.0).sum()
    assert abs(tot[0] - ideal) <= 2e-2 * ideal
