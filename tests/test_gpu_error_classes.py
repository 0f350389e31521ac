"""How a failed cell is reported: a finite energy density that is not positive is an unstable run
(RLBM_E_UNSTABLE) in every storage type and every call that matches the cells, as the header defines
the status."""
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


@pytest.mark.parametrize("call", ["moments", "spectrum", "column_means", "step"])
@pytest.mark.parametrize("precision", ["f64", "f32", "f16", "bf16"])
def test_negative_energy_density_is_unstable(R, precision, call):
    lat = R.Lattice(40, 24, precision=precision, eta_over_s=0.1)
    h, step = lat.get_state()
    h[:, 9:12, 16:19] = -1.5  # the middle cell pulls -1.5 in every class: T^00 = -eps0 / 2, at rest
    lat.set_state(h, step)
    with pytest.raises(R.RlbmError) as e:
        if call == "moments":
            lat.moments()
        elif call == "spectrum":
            lat.spectrum(8)
        elif call == "column_means":
            lat.column_means()
        else:
            lat.step(1)
            lat.sync()
    assert e.value.status == R.RLBM_E_UNSTABLE
    lat.close()
