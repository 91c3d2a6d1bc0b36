"""FP32 grids of more rows than 65,535 tiles of 16 (the most that one dimension
of a launch takes past the first): the tile kernel on a walled one against the
walls sweep, the adjoint tile kernel against the adjoint sweep (which takes
buffers that are only 4-byte aligned)."""
import numpy as np
import pytest

import inputs as I
from conftest import assert_parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_12913_gb300.solver import FDLBM  # noqa: E402

NX, NY = 7, 65_536 * 16 + 5
# twice the FP32 bounds of the step kernels against FP64: both sides are FP32
L2, DEV = 2e-7, 4e-5


def test_tile_step_on_a_tall_walled_grid():
    xa, ya = I.wall_axis(NX - 1, 0.0, 1.0), I.wall_axis(NY - 1, 0.0, 0.25 * (NY - 1))
    wall_u = [(0.0, 0.02), (0.0, -0.01), (0.03, 0.0), (-0.02, 0.0)]
    f = I.random_fields(NX, NY, 5)
    out = {}
    for variant in ("auto", "scalar"):
        s = FDLBM(xa, ya, nu=0.02, cfl=0.3, blend=0.2, precision="fp32", wall_u=wall_u, variant=variant)
        s.init_fields(f["rho"], f["ux"], f["uy"])
        s.step(2)
        s.sync()
        out[variant] = s.get_state()
        kernel = s.describe.split()[0]
        assert kernel == ("fused-tile" if variant == "auto" else "fused-walls"), kernel
        assert s.kernels_per_step == (2 if variant == "auto" else 1)
        s.close()
    assert_parity(out["auto"], out["scalar"], l2=L2, dev=DEV, label=f"{NX}x{NY}")


def test_adjoint_tile_on_a_tall_grid():
    xa, ya = I.periodic_axis(NX, 0.0, 1.0), I.periodic_axis(NY, 0.0, 0.2 * NY)
    s = FDLBM(xa, ya, nu=0.02, cfl=0.4, blend=0.2, adjoint=True, precision="fp32")
    f = I.random_fields(NX, NY, 7)
    s.init_fields(f["rho"], f["ux"], f["uy"])
    gen = torch.Generator(device=s.device).manual_seed(9)
    lam0 = torch.randn((9, NY, s.layout()[0]), generator=gen, device=s.device)
    out = []
    for shift in (0, 1):  # floats past an aligned address
        def buffer():
            return torch.zeros(lam0.numel() + shift, device=s.device)[shift:].view(lam0.shape)
        state, lam, prev = buffer(), buffer(), buffer()
        state.copy_(s.save_state(s.new_buffer()))
        lam.copy_(lam0)
        s.adjoint_step(state, lam, prev)
        s.sync()
        out.append(prev[:, :, :NX].double())
    err = float(torch.linalg.norm(out[0] - out[1]) / torch.linalg.norm(out[1]))
    assert err <= 2e-5, err  # twice the bound of either kernel against FP64
