"""The automatic choice of kernel on both sides of its lines."""
import pytest

import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_12913_gb300.solver import FDLBM  # noqa: E402


def _kernel(nx, ny, *, walls=False, **kw):
    def axis(n):
        return I.wall_axis(n - 1, 0.0, n / 64.0) if walls else I.periodic_axis(n, 0.0, n / 64.0)
    s = FDLBM(axis(nx), axis(ny), nu=0.01, cfl=0.5, blend=0.1, precision="fp32", **kw)
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
