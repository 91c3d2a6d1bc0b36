"""FP32 cavities marched towards their steady state: the tile kernel, the automatic
choice on these grids, settles no further from FP64 than the walls sweep (at a
fixed point every step rounds alike, so a kernel's roundings add up), whichever
wall the lid is on."""
import math

import numpy as np
import pytest

import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_12913_gb300.solver import FDLBM  # noqa: E402

U, RE, STEPS = 0.1, 400.0, 260_000  # E(u) about 1e-9 per step in FP64


@pytest.mark.parametrize("lid", ["N", "E"])
def test_tile_cavity_settles_as_close_to_fp64_as_the_walls_sweep(lid):
    ax = I.tanh_axis(128, 1.5)
    wall_u = [(0, 0), (0, 0), (0, 0), (U, 0.0)] if lid == "N" else [(0, 0), (0, U), (0, 0), (0, 0)]

    def march(**kw):
        s = FDLBM(ax, ax, nu=U / RE, cfl=0.9, blend=0.1, wall_u=wall_u, graph_steps=100, **kw)
        one = np.ones((ax.n, ax.n))
        s.init_fields(one, 0 * one, 0 * one)
        s.step(STEPS)
        s.sync()
        _, ux, uy = s.moments()
        return s.describe.split()[0], np.stack([ux, uy])

    kernel, want = march(precision="fp64")
    assert kernel == "split"
    dist = {}
    for variant in ("auto", "scalar"):
        kernel, u = march(precision="fp32", variant=variant)
        dist[kernel] = math.sqrt(sum((np.linalg.norm(u[k] - want[k]) / np.linalg.norm(want[k])) ** 2 for k in (0, 1)))
    print(lid, dist)
    assert set(dist) == {"fused-tile", "fused-walls"}
    assert dist["fused-tile"] <= dist["fused-walls"]
