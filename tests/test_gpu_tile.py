"""The FP32 tile kernel (step_tile.cu), the automatic choice on small and medium
grids and in FUSED batches, against the oracle: grids smaller than a tile, one
node more or less than whole tiles, widths whose column pairs straddle the
periodic seam or the last wall, walls on one or both axes with moving sides,
random metrics, a force field, the incompressible equilibrium, A = 0, direct
launches and a replayed graph; and the choice itself."""
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

from paper_1911_12913_gb300.solver import FDLBM, FDLBMBatch  # noqa: E402

# The FP32 bounds of the other step kernels over 12 steps from random states.
L2, DEV = 1e-7, 2e-5


def _axis(kind, n, seed, length):
    if kind == "periodic":
        ax = I.periodic_axis(n, 0.0, length)
        ax.metric = I.random_metric(n, seed, base=n / length, spread=0.3)
        return ax
    return I.tanh_axis(n - 1, 1.5) if length == 1.0 else I.wall_axis(n - 1, 0.0, length)


CASES = [
    ("periodic", "periodic", 4, 4, {}), ("periodic", "periodic", 5, 9, {"force": True}),
    ("wall", "wall", 4, 4, {}), ("wall", "wall", 5, 6, {"force": True}),
    ("periodic", "periodic", 33, 17, {"force": True}), ("periodic", "periodic", 31, 15, {}),
    ("periodic", "periodic", 36, 20, {"graph": 4}), ("periodic", "periodic", 131, 70, {"eq": "incompressible"}),
    ("wall", "wall", 33, 17, {}), ("wall", "wall", 34, 18, {"force": True}), ("wall", "wall", 32, 16, {"graph": 2}),
    ("wall", "wall", 65, 33, {"eq": "incompressible", "force": True}), ("wall", "wall", 66, 35, {"A": 0.0}),
    ("periodic", "wall", 100, 40, {"force": True}), ("wall", "periodic", 67, 33, {"eq": "incompressible"}),
    ("periodic", "wall", 37, 50, {}), ("wall", "periodic", 99, 31, {"force": True}),
    ("periodic", "periodic", 128, 128, {"force": True}), ("wall", "wall", 257, 129, {}),
]


def _force(case, rng):
    return 1e-3 * rng.uniform(-1, 1, size=(2, case[3], case[2])) if case[4].get("force") else None


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{c[0][0]}{c[1][0]}-{c[2]}x{c[3]}")
def test_tile_step_matches_oracle(case):
    x, y, nx, ny, more = case
    xa, ya = _axis(x, nx, 31, 1.0), _axis(y, ny, 32, 0.8)
    rng = np.random.default_rng(nx * 1000 + ny)
    force = _force(case, rng)
    wall_u = [tuple(0.05 * rng.uniform(-1, 1, size=2)) for _ in range(4)]
    eq, A = more.get("eq", "standard"), more.get("A", 0.5)
    s = FDLBM(xa, ya, nu=0.02, cfl=0.3, blend=0.2, A=A, precision="fp32", has_force=force is not None,
              wall_u=wall_u, equilibrium=eq, graph_steps=more.get("graph", 0))
    assert s.describe.startswith("fused-tile fp32dev"), s.describe
    assert s.path == "fused" and s.kernels_per_step == 1
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
    assert_parity(s.get_state(), o.f, l2=L2, dev=DEV, label=f"{s.describe} {x}/{y} {nx}x{ny}")


def test_tile_batch_matches_oracle():
    """The same grids in one FUSED batch (every case on the tile kernel: widths
    of 64 and more on a periodic x axis would go to the warp tile)."""
    cases = [c for c in CASES if not (c[0] == "periodic" and c[1] == "periodic" and c[2] >= 64 and c[2] % 4 == 0)]
    probs, args = [], []
    for c in cases:
        x, y, nx, ny, more = c
        rng = np.random.default_rng(nx * 1000 + ny)
        p = dict(xa=_axis(x, nx, 31, 1.0), ya=_axis(y, ny, 32, 0.8), force=_force(c, rng),
                 wall_u=[tuple(0.05 * rng.uniform(-1, 1, size=2)) for _ in range(4)], more=more)
        probs.append(p)
        args.append(dict(xa=p["xa"], ya=p["ya"], nu=0.02, cfl=0.3, blend=0.2, A=more.get("A", 0.5),
                         wall_u=p["wall_u"], has_force=p["force"] is not None,
                         equilibrium=more.get("eq", "standard")))
    b = FDLBMBatch(args, precision="fp32", graph_steps=4, autotune=False)
    assert "warp_tiles=0 " in b.describe and "launches_per_step=1" in b.describe, b.describe
    oracles = []
    for k, (c, p) in enumerate(zip(cases, probs)):
        v = b.case(k)
        o = O.Oracle(p["xa"], p["ya"], nu=0.02, dt=v.dt, beta=0.2, A=p["more"].get("A", 0.5), force=p["force"],
                     wall_u=p["wall_u"], incomp=p["more"].get("eq") == "incompressible")
        if p["force"] is not None:
            v.set_force(p["force"])
        f = I.random_fields(c[2], c[3], 5)
        v.init_fields(f["rho"], f["ux"], f["uy"])
        o.init_fields(f["rho"], f["ux"], f["uy"])
        o.step(12)
        oracles.append(o)
    for n in (5, 7):
        b.step(n)
    b.sync()
    for k, o in enumerate(oracles):
        assert_parity(b.case(k).get_state(), o.f, l2=L2, dev=DEV, label=f"case {k} {cases[k][:4]}")


@pytest.mark.parametrize("x,y,nx,ny,force_on", [
    ("wall", "wall", 1700, 1300, False), ("periodic", "wall", 2048, 1041, True),
    ("wall", "periodic", 1401, 1300, False), ("wall", "wall", 1351, 1413, True), ("wall", "wall", 64, 40000, False)])
def test_warp_tile_with_tile_frame_matches_fp64(x, y, nx, ny, force_on):
    """Large walled grids: the warp tile's interior and the frame on the tile
    kernel store every node once and agree with the FP64 step (checked against
    the oracle elsewhere); east frames of one and two columns of tiles, interiors
    of one window, moving walls, a random force field."""
    xa, ya = _axis(x, nx, 31, 1.0), _axis(y, ny, 32, 0.8)
    rng = np.random.default_rng(nx)
    force = 1e-3 * rng.uniform(-1, 1, size=(2, ny, nx)) if force_on else None
    wall_u = [tuple(0.05 * rng.uniform(-1, 1, size=2)) for _ in range(4)]
    f = I.random_fields(nx, ny, 5)
    out = {}
    for precision in ("fp64", "fp32"):
        s = FDLBM(xa, ya, nu=0.02, cfl=0.3, blend=0.2, precision=precision, has_force=force_on, wall_u=wall_u)
        if force_on:
            s.set_force(force)
        s.init_fields(f["rho"], f["ux"], f["uy"])
        s.step(3)
        s.sync()
        out[precision] = s.get_state()
    assert s.describe.startswith("fused-warp fp32dev") and s.kernels_per_step == 2, s.describe
    assert_parity(out["fp32"], out["fp64"], l2=L2, dev=DEV, label=f"{s.describe} {x}/{y} {nx}x{ny}")


def test_tile_step_is_the_automatic_choice_on_small_and_medium_grids():
    """Each side of the rule's lines, and what keeps the other kernels."""
    def kernel(nx, ny, walls=False, **kw):
        ax = I.wall_axis(nx - 1, 0.0, 1.0) if walls else I.periodic_axis(nx, 0.0, 2 * math.pi)
        ay = I.wall_axis(ny - 1, 0.0, 1.0) if walls else I.periodic_axis(ny, 0.0, 2 * math.pi)
        return FDLBM(ax, ay, nu=0.01, cfl=0.5, blend=0.1, precision="fp32", **kw).describe.split()[0]

    assert kernel(64, 64) == kernel(896, 892) == "fused-tile"
    assert kernel(896, 896) == kernel(300, 33) == "fused-warp"
    assert kernel(1096, 1092, has_force=True) == "fused-tile" and kernel(1100, 1096, has_force=True) == "fused-warp"
    assert kernel(1095, 1095) == "fused-tile" and kernel(1097, 1097) == "fused"
    assert kernel(1117, 1117, walls=True) == "fused-tile" and kernel(1119, 1119, walls=True) == "fused-warp"
    assert kernel(60, 45000, walls=True) == "fused-tile"
    assert kernel(64, 64, variant="warp") == kernel(64, 64, rows_per_cta=4) == kernel(64, 64, path="fused") == "fused-warp"
    assert kernel(33, 33, walls=True, path="fused") == "fused-walls"
    assert kernel(64, 64, scheme=2) == "fused-warp-scheme2"
