"""Batched steps stir with the members' mode multipliers (rlbm_set_mode_scale), set before the batch
was made and between its steps, as steps of the members alone do."""
import os

import numpy as np
import pytest

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


@pytest.mark.parametrize("precision", ["f64", "f32", "f16"])
def test_batch_takes_the_mode_multipliers(R, precision):
    import torch
    stream = torch.cuda.Stream()
    sets = [[R.Lattice(n, 40, stream=stream, precision=precision, eta_over_s=0.05, kmin=2, kmax=5, force_amp=1e-3, seed=n)
             for n in (48, 72)] for _ in range(3)]
    rng = np.random.default_rng(2)
    first, second = (rng.uniform(0.0, 2.0, sets[0][0].num_modes) for _ in range(2))
    alone, batched, plain = sets
    for s in (alone, batched):
        s[0].set_mode_scale(first)
    b, p = R.Batch(batched, stream=stream), R.Batch(plain, stream=stream)
    for steps, sigma in ((3, None), (70, second), (2, np.ones_like(first))):  # (70: a captured chunk too)
        if sigma is not None:
            alone[1].set_mode_scale(sigma)
            batched[1].set_mode_scale(sigma)
        for lat in alone:
            lat.step(steps)
        b.step(steps)
        p.step(steps)
    for k in range(2):
        ma, mb, mp = (s[k].moments() for s in sets)
        for i in range(3):
            assert np.array_equal(ma[i], mb[i])
        assert not np.array_equal(ma[1], mp[1])  # (the multipliers matter)
    for x in [b, p] + alone + batched + plain:
        x.close()
