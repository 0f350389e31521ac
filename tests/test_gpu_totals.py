"""The four totals against sums over the same state: rlbm_get_state's populations pulled once with numpy
in FP64, then T^00, T^0x and T^0y summed over the fluid cells, at shapes where a block sums one tile
and where it sums several.  A cell's FP32 arithmetic takes at most a dozen roundings between the
populations and its moments (weights, four-corner pull, sum over classes), so the totals agree to
12 x 2^-24 < 2^-20 of the sums of absolute terms; FP64 likewise to 2^-49, 2^-47 with the reference's
own roundings, and T^00 to the roundings of its sum of ones, 2^-49 of the number of cells."""
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


def pulled(h, classes, C, solid, walls):
    """Pull-streaming of the planes h: bilinear weights, bounce-back at solid corners."""
    ny, nx = solid.shape
    edge = dict(mode="constant") if walls else dict(mode="wrap")
    blocked = np.pad(np.pad(solid != 0, ((1, 1), (0, 0)), **(dict(edge, constant_values=True) if walls else edge)), ((0, 0), (1, 1)), mode="wrap")
    out = np.empty_like(h)
    for q, (vx, vy, vz2, _) in enumerate(classes):
        opp = int(np.argmin(np.abs(classes[:, 0] + vx) + np.abs(classes[:, 1] + vy) + np.abs(classes[:, 2] - vz2)))
        p = np.pad(np.pad(h[q], ((1, 1), (0, 0)), **edge), ((0, 0), (1, 1)), mode="wrap")
        sx, sy = (int(np.sign(round(v, 9))) for v in (vx, vy))
        ax, ay = C * abs(vx), C * abs(vy)
        out[q] = (1 - ax) * (1 - ay) * h[q]
        for b, ox, oy in ((ax * (1 - ay), sx, 0), ((1 - ax) * ay, 0, sy), (ax * ay, sx, sy)):
            if (ox or oy) and abs(b) > 1e-12:
                sl = (slice(1 - oy, 1 - oy + ny), slice(1 - ox, 1 - ox + nx))
                out[q] += b * np.where(blocked[sl], h[opp], p[sl])
    return out


@pytest.mark.parametrize("precision,tol", [("f64", 2.0 ** -47), ("f32", 2.0 ** -20), ("f16", 2.0 ** -20)])
@pytest.mark.parametrize("nx,ny,walls", [(8, 8, 0), (33, 17, 0), (96, 50, 1), (31, 200, 1), (1200, 500, 0), (1200, 500, 1)])
@pytest.mark.parametrize("vset", [3, 2])
def test_totals_are_the_sums_over_the_state(R, nx, ny, walls, vset, precision, tol):
    e, ux, uy = inputs.smooth_random_fields(nx, ny, seed=7, eps_amp=0.02, u_amp=0.05, kmax=3)
    solid = np.zeros((ny, nx), np.uint8)
    if walls:
        solid[3:9, 5:12] = 1
    lat = R.Lattice(nx, ny, precision=precision, vset=vset, a=0.1, dt=0.05, eta_over_s=0.1, walls_y=walls, solid=solid if walls else None,
                    eps0=1.25, init_eps=1.25 * 1.05 * e, init_ux=ux + 0.02, init_uy=uy - 0.01)
    lat.step(3)
    h, _ = lat.get_state()
    tot = lat.totals()
    lat.close()
    cl = R.rlbm_velocity_classes(vset)
    fluid = solid == 0
    f = pulled(h, cl, 0.5, solid, walls)[:, fluid]
    for k, v in enumerate((np.ones(len(cl)), cl[:, 0], cl[:, 1])):
        t = (cl[:, 3] * v)[:, None] * f
        want = 1.25 * (t.sum() + (fluid.sum() if k == 0 else 0))
        assert abs(tot[k] - want) <= 1.25 * (tol * np.abs(t).sum() + (fluid.sum() * 2.0 ** -49 if k == 0 else 0.0)), (k, tot[k], want)
