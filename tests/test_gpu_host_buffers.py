"""The small results of a context come to the host through a buffer that rlbm_init allocates: calls that
read them allocate nothing of their size (an allocation that fails there would throw through the C
ABI).  Counted by the C library: blocks above its mmap threshold (128 KB at the start)."""
import ctypes
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


class Mallinfo2(ctypes.Structure):
    _fields_ = [(n, ctypes.c_size_t) for n in ("arena", "ordblks", "smblks", "hblks", "hblkhd", "usmblks", "fsmblks", "uordblks", "fordblks", "keepcost")]


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


def test_reading_small_results_allocates_no_large_block(R):
    libc = ctypes.CDLL(None)
    if not hasattr(libc, "mallinfo2"):
        pytest.skip("no mallinfo2")
    libc.mallinfo2.restype = Mallinfo2
    used = lambda: (lambda m: m.hblkhd + m.uordblks)(libc.mallinfo2())  # noqa: E731
    nx = 16384  # column means: 2 x 128 KB
    warm = R.Lattice(64, 8)
    for call in (warm.totals, warm.column_means):  # the runtime's own first allocations
        call()
    lat = R.Lattice(nx, 8)
    jx, jy = np.empty(nx), np.empty(nx)
    lat.totals()
    before = used()
    R.rlbm_column_means(lat.ctx, jx, jy)
    after = used()
    assert after - before < 16 * nx // 2, (before, after)
    lat.close()
    warm.close()
