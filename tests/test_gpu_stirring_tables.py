"""Stirring tables at the edges of their construction, against the oracle: rows longer than one
warp's chunk (256 columns in FP32, 128 in FP64) with a ragged last chunk, rows of more than 32
modes, shells of more than 16 rows (read from global memory, not staged), and lattices with a CTA
for every tile and table chunk as well as far more of them than CTAs.  FP64 1e-10, FP32 1e-5 in
eps (relative) and u (relative to max |u|), the bars of the other parity tests."""
import os

import numpy as np
import pytest

from oracle import rlbm_oracle as O
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


@pytest.mark.parametrize("nx,ny,kmin,kmax", [(130, 16, 2, 4), (257, 24, 3, 5), (515, 16, 1, 6), (48, 41, 0, 19), (300, 260, 8, 10)])
@pytest.mark.parametrize("precision,tol", [("f64", 1e-10), ("f32", 1e-5)])
def test_stirred_run_matches_the_oracle(R, nx, ny, kmin, kmax, precision, tol):
    e, ux, uy = inputs.smooth_random_fields(nx, ny, seed=nx, u_amp=0.02, kmax=3)
    cfg = dict(nx=nx, ny=ny, eta_over_s=0.05, kmin=kmin, kmax=kmax, force_amp=1e-3, seed=5,
               init_eps=e, init_ux=ux, init_uy=uy)
    ref = O.run(cfg, 4)
    lat = R.Lattice(nx, ny, precision=precision, **{k: v for k, v in cfg.items() if k not in ("nx", "ny")})
    lat.step(1)
    lat.step(3)
    got = lat.moments()
    lat.close()
    umax = max(np.abs(ref[1]).max(), np.abs(ref[2]).max())
    assert np.max(np.abs(got[0] - ref[0]) / ref[0]) <= tol
    assert max(np.abs(got[1] - ref[1]).max(), np.abs(got[2] - ref[2]).max()) <= tol * umax
