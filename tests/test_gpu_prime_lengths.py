"""Transforms whose length is a prime number: a direct sum per output, the same work along x as along y,
so a lattice and its transpose take about the same time; their spectra agree to rounding."""
import os
import time

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


@pytest.mark.parametrize("few,prime", [(64, 2039), (127, 1021)])
def test_a_prime_length_costs_the_same_along_x_and_y(R, few, prime):
    """FP64 (64 x 2039 took 22.7 ms and 2039 x 64 took 11.4 ms with two columns to a block)."""
    rng = np.random.default_rng(3)
    ux, uy = (1e-2 * rng.standard_normal((prime, few)) for _ in range(2))
    ms, E = {}, {}
    for name, shape, u, v in (("y", (few, prime), ux, uy), ("x", (prime, few), uy.T, ux.T)):
        lat = R.Lattice(*shape, precision="f64", init_ux=u, init_uy=v)
        E[name] = lat.spectrum(40)
        times = []
        for _ in range(5):
            t = time.perf_counter()
            lat.spectrum(40)
            times.append(time.perf_counter() - t)
        ms[name] = 1e3 * min(times)
        lat.close()
    print(ms)
    assert np.abs(E["x"] - E["y"]).max() <= 1e-12 * E["x"].max()
    assert ms["y"] <= 1.4 * ms["x"], ms
