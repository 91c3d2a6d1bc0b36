"""Total momentum of a periodic flow on the FP64 split step: conserved by the
scheme, so that only roundings move it.  Roundings that do not lean to one side
average out over 37,000 nodes; a lean of 1 % of an FP64 rounding per step
(1e-18) shows as 1e-15 after 1000 steps."""
import math

import numpy as np
import pytest

import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_12913_gb300.solver import FDLBM  # noqa: E402


@pytest.mark.parametrize("n", [64, 192])  # four threads per node, one thread per node
def test_split_step_does_not_lean(n):
    ax = I.periodic_axis(n, 0.0, 2 * math.pi)
    f = I.taylor_green(ax, ax, u0=0.05)
    s = FDLBM(ax, ax, nu=0.001, cfl=0.5, blend=0.1)
    assert s.describe.startswith("split fp64")
    s.init_fields(f["rho"], f["ux"] + 0.05, f["uy"] + 0.02, [f["dudx"], f["dudy"], f["dvdx"], f["dvdy"]])

    def momentum():
        g = s.get_state()
        g -= np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4).reshape(9, 1, 1)
        total = lambda i: math.fsum(g[i].ravel())  # noqa: E731
        return (total(1) - total(3) + total(5) - total(6) - total(7) + total(8),
                total(2) - total(4) + total(5) + total(6) - total(7) - total(8))

    j0 = momentum()
    s.step(1000)
    j1 = momentum()
    drift = [abs(b / a - 1.0) for a, b in zip(j0, j1)]
    print(n, drift)
    assert max(drift) <= 3e-15
