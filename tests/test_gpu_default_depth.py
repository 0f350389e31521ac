"""The default pipeline depth of a form is the faster one, or within 3.5 % of it, at 2048 x 512 (the forms
whose depths differ by 5 %: 16-bit and FP32 storage between walls, with and without a body force)."""
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
@pytest.mark.parametrize("force", ["none", "body", "stirred"])
def test_default_depth_is_the_faster(R, precision, force):
    import torch
    nx, ny = 2048, 512
    stream = torch.cuda.Stream()
    mask, _ = inputs.disc_mask(nx, ny, radius=6, fraction=0.05, seed=1, walls_y=force != "stirred")
    kw = {"none": dict(walls_y=1), "body": dict(walls_y=1, body_force=(1e-6, 0.0)), "stirred": dict(kmin=4, kmax=6, force_amp=1e-5)}[force]
    us = {}
    for stages in (0, 1, 2):
        lat = R.Lattice(nx, ny, stream=stream, precision=precision, eta_over_s=0.05, solid=np.asarray(mask, np.uint8), **kw)
        if stages:
            lat.set_launch(0, stages)
        times = []
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            lat.step(200)
            b.record(stream)
            lat.sync()
            times.append(a.elapsed_time(b) * 5.0)
        us[stages] = min(times)
        lat.close()
    print(us)
    assert us[0] <= 1.035 * min(us[1], us[2]), us
