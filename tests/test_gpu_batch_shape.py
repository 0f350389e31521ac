"""The pipeline depth of a batch: the one set on its first member before the batch was made, until one is
set on the batch.  Results do not tell depths apart; their times do (FP32 without a mask: two stages
are a tenth slower), so the batch's own time is compared with that of either depth."""
import os

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


def test_a_depth_set_on_the_members_stays(R):
    import torch
    stream = torch.cuda.Stream()

    def us(batch):
        times = []
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            batch.step(128)
            b.record(stream)
            b.synchronize()
            times.append(a.elapsed_time(b) / 0.128)
        return min(times)

    lats = [R.Lattice(512, 512, stream=stream, precision="f32", eta_over_s=0.05, kmin=8, kmax=10, force_amp=1e-5, seed=i) for i in range(16)]
    b = R.Batch(lats, stream=stream)
    one = us(b)  # the default of this form
    b.set_launch(0, 2)
    two = us(b)
    b.close()
    lats[0].set_launch(0, 2)
    b = R.Batch(lats, stream=stream)
    kept = us(b)
    b.set_launch(0, 1)
    again = us(b)
    print("one stage %.1f us, two %.1f, two set on the member %.1f, one set on the batch %.1f" % (one, two, kept, again))
    assert two > 1.03 * one  # (else the comparison says nothing)
    assert abs(kept - two) < abs(kept - one)
    assert abs(again - one) < abs(again - two)
    b.close()
    for lat in lats:
        lat.close()
