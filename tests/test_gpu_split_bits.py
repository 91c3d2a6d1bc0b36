"""Bits of the FP64 split step: the same from run to run, where four threads of a
node read what one of them then overwrites in place; and the same however the
steps are divided into calls or replayed from a graph, so that a run can be
stopped and resumed."""
import numpy as np
import pytest

import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_12913_gb300.solver import FDLBM  # noqa: E402


def _axis(kind, n, seed, length):
    if kind == "periodic":
        ax = I.periodic_axis(n, 0.0, length)
        ax.metric = I.random_metric(n, seed, base=n / length, spread=0.3)
        return ax
    return I.tanh_axis(n - 1, 1.5)


def _solver(x, y, nx, ny, force, **kw):
    s = FDLBM(_axis(x, nx, 1, 1.0), _axis(y, ny, 2, 0.8), nu=0.02, cfl=0.3, blend=0.2, has_force=force,
              wall_u=[(0, 0.01), (0, 0.02), (0.03, 0), (-0.01, 0)], **kw)
    assert s.describe.startswith("split fp64")
    if force:
        s.set_force(1e-3 * np.random.default_rng(3).uniform(-1, 1, size=(2, ny, nx)))
    f = I.random_fields(nx, ny, 5)
    s.init_fields(f["rho"], f["ux"], f["uy"])
    return s


@pytest.mark.parametrize("nx,ny,force", [(3, 3, False), (33, 17, True), (64, 64, False), (97, 100, True)])
def test_in_place_quads_give_the_same_bits_every_time(nx, ny, force):
    states = [_solver("periodic", "periodic", nx, ny, force).step(100).get_state() for _ in range(3)]
    assert np.array_equal(states[0], states[1]) and np.array_equal(states[0], states[2])


@pytest.mark.parametrize("x,y,nx,ny,force", [
    ("periodic", "periodic", 64, 64, False), ("periodic", "periodic", 33, 17, True),
    ("periodic", "periodic", 160, 129, False), ("periodic", "periodic", 160, 129, True),
    ("wall", "wall", 33, 33, False), ("wall", "wall", 40, 30, True), ("wall", "wall", 129, 97, False),
    ("wall", "wall", 129, 97, True), ("periodic", "wall", 150, 70, True), ("wall", "periodic", 150, 70, False),
])
def test_state_does_not_depend_on_the_division_into_calls(x, y, nx, ny, force):
    whole = _solver(x, y, nx, ny, force).step(24).get_state()
    s = _solver(x, y, nx, ny, force)
    for n in (1, 1, 2, 5, 1, 14):
        s.step(n)
    assert np.array_equal(s.get_state(), whole)
    assert np.array_equal(_solver(x, y, nx, ny, force, graph_steps=4).step(24).get_state(), whole)
    # resumed from a saved state
    s = _solver(x, y, nx, ny, force).step(10)
    kept = s.save_state(s.new_buffer())
    s.step(3)
    assert np.array_equal(s.load_state(kept).step(14).get_state(), whole)
