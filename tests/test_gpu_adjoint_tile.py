"""The FP32 adjoint tile kernel (adjoint_tile.cu) against the FP64 adjoint sweep
(itself checked against the transposed Jacobian of the oracle's step): grids
smaller than a tile, one node more or less than whole tiles, odd widths (column
pairs across the periodic seam), with and without a force field and a force
cotangent, and buffers that are only 4-byte aligned, which keep the sweep."""
import numpy as np
import pytest

import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_12913_gb300.solver import FDLBM  # noqa: E402


def _rel(a, b):
    return float(torch.linalg.norm(a.double() - b) / torch.linalg.norm(b))


def _step(precision, nx, ny, force_on, df_on, shift=0):
    xa, ya = I.periodic_axis(nx, 0.0, 1.0), I.periodic_axis(ny, 0.0, 0.9)
    xa.metric = I.random_metric(nx, 1, base=nx, spread=0.3)
    ya.metric = I.random_metric(ny, 2, base=ny / 0.9, spread=0.3)
    s = FDLBM(xa, ya, nu=0.02, cfl=0.4, blend=0.2, has_force=force_on, adjoint=True, precision=precision)
    rng = np.random.default_rng(nx * 1000 + ny)
    if force_on:
        s.set_force(2e-3 * rng.uniform(-1, 1, size=(2, ny, nx)))
    f = I.random_fields(nx, ny, 7)
    s.init_fields(f["rho"], f["ux"], f["uy"], [f["dudx"], f["dudy"], f["dvdx"], f["dvdy"]])

    def buffer():  # `shift` floats past an aligned address
        b = s.new_buffer()
        return torch.zeros(b.numel() + shift, dtype=b.dtype, device=b.device)[shift:].view(b.shape)

    state, lam, out = buffer(), buffer(), buffer()
    state.copy_(s.save_state(s.new_buffer()))
    lam[:, :, :nx] = torch.as_tensor(np.random.default_rng(9).normal(size=(9, ny, nx)), dtype=lam.dtype)
    dF = torch.ones((2, ny, nx), dtype=torch.float64, device=s.device) if df_on else None
    s.adjoint_step(state, lam, out, dF)
    s.sync()
    assert not out[:, :, nx:].any()  # the padding stays as it was
    return out[:, :, :nx], dF


@pytest.mark.parametrize("nx,ny,force_on,df_on,shift", [
    (4, 4, True, True, 0), (5, 9, True, True, 0), (31, 15, True, True, 0), (32, 16, False, True, 0),
    (33, 17, True, True, 0), (36, 20, True, False, 0), (64, 48, True, True, 0), (67, 33, False, True, 0),
    (131, 50, True, True, 0), (256, 40, False, False, 0), (64, 32, True, True, 1), (33, 17, True, True, 1),
])
def test_adjoint_tile_matches_fp64(nx, ny, force_on, df_on, shift):
    """One step: the rounding of a sum of some hundred FP32 products of O(1)
    cotangents, 1e-7 relative; bounds of the sweep's own FP32 test."""
    want, wF = _step("fp64", nx, ny, force_on, df_on)
    got, gF = _step("fp32", nx, ny, force_on, df_on, shift)
    assert _rel(got, want) <= 1e-5
    if df_on:
        assert _rel(gF - 1.0, wF - 1.0) <= 1e-4
