"""The FP64 step in two launches (step_split.cu), the automatic choice and
path="staged", against the oracle (four threads per node on
small FP64 grids and at FP64 wall nodes): strips of one column
to several, partial last warps and strips, grids of three nodes per axis, every
boundary combination with moving walls, random metrics, a force field, the
incompressible equilibrium, A = 0, direct launches and a replayed graph."""
import math

import numpy as np
import pytest

import inputs as I
import oracle as O
from conftest import assert_parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_12913_gb300.solver import FDLBM  # noqa: E402

# The bounds of the other FP64 step kernels: 12 steps of O(1e-16) roundings, with
# the margin used there.
L2, DEV = 1e-12, 1e-11


def _axis(kind, n, seed, length):
    if kind == "periodic":
        ax = I.periodic_axis(n, 0.0, length)
        ax.metric = I.random_metric(n, seed, base=n / length, spread=0.3)
        return ax
    return I.tanh_axis(n - 1, 1.5) if length == 1.0 else I.wall_axis(n - 1, 0.0, length)


@pytest.mark.parametrize("path", ["auto", "staged"])
@pytest.mark.parametrize("x,y,nx,ny,more", [
    ("periodic", "periodic", 3, 3, {}), ("wall", "wall", 3, 3, {}), ("wall", "periodic", 3, 7, {}),
    ("periodic", "wall", 4, 3, {}), ("periodic", "periodic", 31, 33, {"force": True}),
    ("periodic", "periodic", 65, 5, {"graph": 4}), ("wall", "wall", 66, 67, {"graph": 4}),
    ("wall", "wall", 131, 9, {"force": True}), ("periodic", "wall", 130, 34, {"force": True, "graph": 2}),
    ("wall", "periodic", 67, 40, {"eq": "incompressible", "force": True}),
    ("periodic", "periodic", 96, 40, {"eq": "incompressible"}), ("periodic", "wall", 64, 20, {"A": 0.0}),
    # FP64 grids past the sizes that take four threads per node throughout
    ("wall", "wall", 257, 40, {}), ("periodic", "periodic", 200, 129, {}), ("periodic", "periodic", 160, 64, {"force": True}),
    ("wall", "wall", 131, 80, {"force": True, "graph": 2}), ("periodic", "wall", 150, 70, {"force": True}),
    ("wall", "periodic", 140, 90, {"eq": "incompressible", "force": True}), ("wall", "wall", 99, 98, {"A": 0.0}),
    # and on both sides of those lines
    ("periodic", "periodic", 128, 76, {}), ("periodic", "periodic", 139, 70, {}), ("wall", "wall", 76, 64, {}),
    ("wall", "wall", 65, 75, {}),
])
def test_split_step_matches_oracle(path, x, y, nx, ny, more):
    xa, ya = _axis(x, nx, 31, 1.0), _axis(y, ny, 32, 0.8)
    rng = np.random.default_rng(nx * 1000 + ny)
    force = 1e-3 * rng.uniform(-1, 1, size=(2, ny, nx)) if more.get("force") else None
    wall_u = [tuple(0.05 * rng.uniform(-1, 1, size=2)) for _ in range(4)]
    eq, A = more.get("eq", "standard"), more.get("A", 0.5)
    s = FDLBM(xa, ya, nu=0.02, cfl=0.3, blend=0.2, A=A, has_force=force is not None,
              wall_u=wall_u, equilibrium=eq, path=path, graph_steps=more.get("graph", 0))
    assert s.describe.startswith("split fp64"), s.describe
    assert s.kernels_per_step == 2
    o = O.Oracle(xa, ya, nu=0.02, dt=s.dt, beta=0.2, A=A, force=force, wall_u=wall_u,
                 incomp=eq == "incompressible")
    if force is not None:
        s.set_force(force)
    f = I.random_fields(nx, ny, 5)
    grad = [f["dudx"], f["dudy"], f["dvdx"], f["dvdy"]]
    s.init_fields(f["rho"], f["ux"], f["uy"], grad)
    o.init_fields(f["rho"], f["ux"], f["uy"], grad)
    for n in (1, 0, 11):
        s.step(n)
        o.step(n)
    s.sync()
    assert s.steps_done == 12
    assert_parity(s.get_state(), o.f, l2=L2, dev=DEV, label=f"{s.describe} {x}/{y} {nx}x{ny}")


def test_split_step_is_the_automatic_choice_for_fp64_only():
    """A tile height or a kernel that is asked for, and T2S2-FDLBM2, keep the
    sweeps and the staged kernels; so does FP32."""
    pa, wa = I.periodic_axis(64, 0.0, 2 * math.pi), I.wall_axis(20, 0.0, 1.0)
    kw = dict(nu=0.01, cfl=0.5, blend=0.1)
    assert FDLBM(pa, pa, **kw).path == "fused"
    assert FDLBM(wa, wa, **kw).path == "staged"
    assert FDLBM(pa, pa, rows_per_cta=4, **kw).describe.startswith("fused fp64")
    assert FDLBM(pa, pa, variant="scalar", **kw).describe.startswith("fused fp64")
    assert FDLBM(pa, pa, path="fused", **kw).describe.startswith("fused fp64")
    assert FDLBM(pa, pa, scheme=2, **kw).describe.startswith("fused-scheme2")
    assert not FDLBM(pa, pa, precision="fp32", **kw).describe.startswith("split")
    assert FDLBM(wa, wa, precision="fp32", path="staged", **kw).describe.startswith("staged fp32dev")
