"""The tile height that a batch's tuning keeps for later batches of the same
grids: it belongs to the kernels that the cases run on."""
import re

import pytest

import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_12913_gb300.solver import FDLBMBatch  # noqa: E402


def _rows(variant, autotune=True):
    ax = I.tanh_axis(511, 1.5)
    cases = [dict(xa=ax, ya=ax, nu=1e-3, cfl=0.9, blend=0.1, variant=variant) for _ in range(6)]
    b = FDLBMBatch(cases, precision="fp32", graph_steps=10, autotune=autotune)
    d = b.describe
    b.close()
    return int(re.search(r"rows=(\d+)", d).group(1)), "warp_tiles=0 " not in d


def test_tuned_height_is_not_taken_over_from_another_kernel():
    """A batch on the tile kernel, which has no height, then one of the same grids
    on the warp tile: 6 x 10 windows of 512 rows fill 1,216 slots at 26 rows or so,
    and the tuning tries a half to twice of what the model says."""
    model, warp = _rows("warp", autotune=False)
    assert warp and model >= 16
    rows, warp = _rows("auto")
    assert not warp and rows > 1  # no height of its own: not the smallest, which suits no sweep
    rows, warp = _rows("warp")
    assert warp and model // 2 <= rows <= 2 * model, (rows, model)
