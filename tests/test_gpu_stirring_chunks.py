"""A row of the stirring table is built in chunks of columns, one warp each: lattices whose width is at
the edge of a chunk of 64 columns (FP32) or 128 (FP64), against the oracle (FP64 1e-10, FP32 1e-5 in eps
(relative) and u (relative to max |u|), the bars of the other parity tests), and the time that a shell
of many modes adds to a small lattice's step."""
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


@pytest.mark.parametrize("nx", [31, 63, 64, 65, 127, 128, 129])
@pytest.mark.parametrize("precision,tol", [("f64", 1e-10), ("f32", 1e-5)])
def test_rows_at_the_edges_of_chunks(R, nx, precision, tol):
    e, ux, uy = inputs.smooth_random_fields(nx, 27, seed=nx, u_amp=0.02, kmax=3)
    cfg = dict(nx=nx, ny=27, eta_over_s=0.05, kmin=6, kmax=12, force_amp=1e-3, seed=5, init_eps=e, init_ux=ux, init_uy=uy)
    ref = O.run(cfg, 3)
    lat = R.Lattice(nx, 27, precision=precision, **{k: v for k, v in cfg.items() if k not in ("nx", "ny")})
    lat.step(3)
    got = lat.moments()
    lat.close()
    umax = max(np.abs(ref[1]).max(), np.abs(ref[2]).max())
    assert np.max(np.abs(got[0] - ref[0]) / ref[0]) <= tol
    assert max(np.abs(got[1] - ref[1]).max(), np.abs(got[2] - ref[2]).max()) <= tol * umax


def test_a_shell_of_many_modes_does_not_set_the_step_time(R):
    """128^2: building the rows of 166 modes hides behind the step's other work, as that of 20 modes
    does (3.7 and 5.1 us per step; 4.0 and 7.1 with chunks of 256 columns)."""
    import torch
    stream = torch.cuda.Stream()
    us = {}
    for shell in ((2, 4), (6, 12)):
        lat = R.Lattice(128, 128, stream=stream, precision="f32", eta_over_s=0.05, kmin=shell[0], kmax=shell[1], force_amp=1e-5, seed=3)
        times = []
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            lat.step(500)
            b.record(stream)
            lat.sync()
            times.append(a.elapsed_time(b) * 2.0)
        us[shell] = min(times)
        lat.close()
    print(us)
    assert us[6, 12] <= 1.5 * us[2, 4], us
