"""Lattices whose two buffers no longer fit in L2 walk their tiles backwards on odd steps; the batch
never does.  A run of both kinds of steps, alone with one and with two tiles of shared memory and as a
batch of one member, gives the same bits: every cell is computed the same way whatever the order."""
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


@pytest.mark.parametrize("precision,nx,ny", [("f32", 901, 853), ("f16", 1283, 1181), ("f64", 643, 599)])
@pytest.mark.parametrize("masked", [False, True])
def test_large_lattices_step_alike_in_either_order(R, precision, nx, ny, masked):
    e, ux, uy = inputs.smooth_random_fields(nx, ny, seed=3, u_amp=0.02, kmax=3)
    mask = None
    if masked:
        mask = np.zeros((ny, nx), np.uint8)
        mask[200:217, 130:171] = 1
        mask[ny - 1, nx - 1] = mask[0, 0] = 1

    def make():
        return R.Lattice(nx, ny, precision=precision, eta_over_s=0.05, kmin=4, kmax=6, force_amp=1e-4, seed=9,
                         init_eps=e, init_ux=ux, init_uy=uy, solid=mask)

    one, two, member = make(), make(), make()
    two.set_launch(0, 3 - (2 if precision == "f16" else 1))
    batch = R.Batch([member])
    for n in (1, 2):
        one.step(n)
        two.step(n)
        batch.step(n)
    want = member.moments()
    for lat in (one, two):
        for a, b in zip(lat.moments(), want):
            assert np.array_equal(np.asarray(a), np.asarray(b))
    batch.close()
    for lat in (one, two, member):
        lat.close()
