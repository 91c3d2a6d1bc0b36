"""The automatic choice of kernel on both sides of its lines."""
import numpy as np
import pytest

import inputs as I
from conftest import assert_parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_12913_gb300.solver import FDLBM  # noqa: E402


def _axis(n, walls):
    return I.wall_axis(n - 1, 0.0, n / 64.0) if walls else I.periodic_axis(n, 0.0, n / 64.0)


def _kernel(nx, ny, *, walls=False, **kw):
    s = FDLBM(_axis(nx, walls), _axis(ny, walls), nu=0.01, cfl=0.5, blend=0.1, precision="fp32", **kw)
    kernel = s.describe.split()[0]
    s.close()
    return kernel


@pytest.mark.parametrize("force", [False, True])
def test_walled_scheme2_has_a_line_of_its_own(force):
    """T2S2-FDLBM2 has no tile kernel: its walled grids change from the walls
    sweep to the warp tile where those two cross, at the same size with and
    without a force, and later on thin grids, which are mostly frame."""
    for nx, ny, want in ((1117, 1117, "fused-scheme2"), (1119, 1119, "fused-warp-scheme2"),
                         (1300, 1300, "fused-warp-scheme2"), (100, 14000, "fused-scheme2"),
                         (14000, 100, "fused-scheme2"), (100, 16000, "fused-warp-scheme2")):
        assert _kernel(nx, ny, walls=True, scheme=2, has_force=force) == want, (nx, ny, force)


def test_tile_kernel_on_small_grids_and_not_on_thin_large_ones():
    """Periodic grids: small ones take the tile kernel, whatever part of their tiles
    they fill (thin ones from 0.65 on); where a grid of many tiles fills them badly, the
    warp tile or the scalar sweep is faster and keeps it."""
    for nx, ny in ((68, 68), (64, 17), (72, 72), (100, 100), (64, 33), (128, 33), (200, 50), (580, 1000), (33, 30000), (1001, 1001)):
        assert _kernel(nx, ny) == _kernel(nx, ny, has_force=True) == "fused-tile", (nx, ny)
    for nx, ny in ((100, 7000), (20000, 33)):
        assert _kernel(nx, ny) == _kernel(nx, ny, has_force=True) == "fused-warp", (nx, ny)
    for nx, ny in ((772, 1000), (196, 3500)):
        assert _kernel(nx, ny) == "fused-warp" and _kernel(nx, ny, has_force=True) == "fused-tile", (nx, ny)
    assert _kernel(30001, 33) == _kernel(30001, 33, has_force=True) == "fused"


def test_thin_walled_grids_stay_on_the_tile_kernel_longer():
    for nx, ny in ((66, 20000), (20000, 66), (100, 15700)):
        assert _kernel(nx, ny, walls=True) == _kernel(nx, ny, walls=True, has_force=True) == "fused-tile", (nx, ny)
    assert _kernel(66, 24000, walls=True) == "fused-warp" and _kernel(300, 4400, walls=True) == "fused-warp"
    assert _kernel(66, 24000, walls=True, has_force=True) == "fused-tile"


@pytest.mark.parametrize("ny,force", [(66, False), (179, False), (180, False), (66, True), (111, True), (112, True)])
def test_frame_of_a_channel_of_few_rows_is_a_walls_sweep(ny, force):
    """Walls in y only: few rows keep the frame that variant="warp" runs (the same
    bits), more rows take the tile kernel's (other roundings); both agree."""
    nx = 1_700_000 // ny // 4 * 4 + 8
    rng = np.random.default_rng(ny)
    f = I.random_fields(nx, ny, 5)
    F = 1e-3 * rng.uniform(-1, 1, size=(2, ny, nx)) if force else None
    out = []
    for variant in ("auto", "warp"):
        s = FDLBM(_axis(nx, False), _axis(ny, True), nu=0.02, cfl=0.3, blend=0.2, precision="fp32", has_force=force,
                  variant=variant, wall_u=[(0, 0), (0, 0), (0.02, 0), (-0.03, 0)])
        assert s.describe.split()[0] == "fused-warp"
        if force:
            s.set_force(F)
        s.init_fields(f["rho"], f["ux"], f["uy"])
        s.step(3)
        out.append(s.get_state())
        s.close()
    assert np.array_equal(out[0], out[1]) == (ny < (112 if force else 180))
    assert_parity(out[0], out[1], l2=2e-7, dev=4e-5, label=f"{nx}x{ny}")  # both sides FP32: twice their bound against FP64
