"""Every storage type, with and without a mask, stepped with one and with two tiles of shared memory, by
default and as a batch of either depth: the same bits."""
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


@pytest.mark.parametrize("nx,ny", [(70, 45), (421, 333)])
@pytest.mark.parametrize("precision", ["f32", "f16", "bf16", "f64"])
@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("force", ["none", "stirred"])
def test_one_and_two_stages_give_the_same_bits(R, precision, masked, force, nx, ny):
    e, ux, uy = inputs.smooth_random_fields(nx, ny, seed=3, u_amp=0.02, kmax=3)
    mask = None
    if masked:
        mask = np.zeros((ny, nx), np.uint8)
        mask[20:37, 13:41] = 1
        mask[ny - 1, nx - 1] = mask[0, 0] = 1
    kw = dict(kmin=4, kmax=6, force_amp=1e-4, seed=9) if force == "stirred" else {}

    def make(stages=0):
        lat = R.Lattice(nx, ny, precision=precision, eta_over_s=0.05, init_eps=e, init_ux=ux, init_uy=uy, solid=mask, **kw)
        if stages:
            lat.set_launch(0, stages)
        return lat

    alone = [make(s) for s in (0, 1, 2)]
    members = [make(), make()]
    batches = [R.Batch([m]) for m in members]
    for b, s in zip(batches, (1, 2)):
        b.set_launch(0, s)
    for n in (1, 4):
        for x in alone + batches:
            x.step(n)
    want = alone[0].moments()
    for lat in alone[1:] + members:
        for a, b in zip(lat.moments()[:3], want[:3]):
            assert np.array_equal(a, b)
    for x in batches + alone + members:
        x.close()
