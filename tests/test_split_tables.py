"""The difference weights of the FP64 split step (host-side, no GPU): the rounded
weights of each node and sign, with the metric and the time step folded in, sum
to exactly zero, so that no step scales a population, and give a linear function
its slope, so that populations travel at their speed; each lies within its grid
of the exact product; and the centre weights of the two axes count as merged only
where their sum is exact.  Checked in rational arithmetic on hex floats that a
small host program built from the CUDA sources prints."""
import os
import shutil
import subprocess
from fractions import Fraction as Fr
from pathlib import Path

import numpy as np
import pytest

import inputs as I

ROOT = Path(__file__).resolve().parents[1]
CSRC = ROOT / "paper_1911_12913_gb300" / "csrc"


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or (os.path.exists("/usr/local/cuda/bin/nvcc") and "/usr/local/cuda/bin/nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    exe = tmp_path_factory.mktemp("st") / "split_tables"
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "-I", str(CSRC),
                    "-I", str(ROOT / "include"), "-o", str(exe), str(ROOT / "tests" / "native" / "split_tables.cu")],
                   check=True, capture_output=True)
    return exe


def _tables(program, beta, wx, wy, h, dt, mx, my):
    args = [repr(float(beta)), str(int(wx)), str(int(wy)), repr(float(h)), repr(float(dt)), str(len(mx))]
    out = subprocess.run([str(program), *args, *(repr(float(v)) for v in (*mx, *my))], check=True,
                         capture_output=True, text=True).stdout.splitlines()
    return out[0] == "merge 1", [[Fr(float.fromhex(v)) for v in line.split()] for line in out[1:]]


def _cases():
    rng = np.random.default_rng(7)
    for beta in (0.0, 0.1, 0.3, 0.31, 0.7, 1.0):
        yield beta, False, False, 2e-3, 4e-3, np.full(5, 64 / (2 * np.pi)), np.full(4, 64 / (2 * np.pi))
        yield beta, False, False, 3e-4, 6e-4, I.random_metric(7, 1, base=50.0, spread=0.3), I.random_metric(6, 2, base=7e3,
                                                                                                      spread=0.3)
        ax = I.tanh_axis(16, 1.5)
        yield beta, True, True, 5.3e-4, 1.06e-3, ax.metric, I.wall_axis(9, 0.0, 0.7).metric
        yield beta, True, False, 0.0, 1.06e-3, ax.metric, np.exp(rng.uniform(-8, 8, size=6))


def test_split_weights_keep_sum_and_slope(program):
    for beta, wx, wy, h, dt, mx, my in _cases():
        merge, rows = _tables(program, beta, wx, wy, h, dt, mx, my)
        b = Fr(float(beta))
        mixed = [(1 - b) / 2, 3 * b / 2, -(1 - b) / 2 - 2 * b, b / 2]
        at, centres = 0, {}
        for name, m, wall, s in (("bx", mx, wx, h), ("by", my, wy, h), ("cx", mx, wx, dt), ("cy", my, wy, dt)):
            for k in range(len(m)):
                for sign in (1, -1):
                    w = rows[at]
                    at += 1
                    assert sum(w) == 0, (beta, name, k, sign)
                    central = wall and (k < 2 if sign > 0 else k > len(m) - 3)
                    scale = -Fr(float(s)) * Fr(float(m[k]))
                    ulp = abs(scale) / 2 ** 52
                    # the slope: the FP64 rounding of the product (half an ulp), and the grid of
                    # two ulps that a blend above 0.3 needs (one more)
                    assert abs(w[0] - w[2] - 2 * w[3] - scale) <= (ulp / 2 if beta <= 0.3 or central else 3 * ulp / 2)
                    # m1 and p2: half their grid (one ulp), their own rounding and that of scale
                    # (one ulp); the other two take up twice their errors and the slope's
                    exact = [scale * v for v in ([Fr(1, 2), 0, Fr(-1, 2), 0] if central else mixed)]
                    assert max(abs(a - e) for a, e in zip(w, exact)) <= 8 * ulp, (beta, name, k, sign)
                    centres.setdefault(name, set()).add(w[1])
        assert at == len(rows)
        if merge:
            for x, y in (("bx", "by"), ("cx", "cy")):
                assert len(centres[x]) == len(centres[y]) == 1
                (a,), (c,) = centres[x], centres[y]
                assert Fr(float(a) + float(c)) == a + c
        # the common case, a uniform periodic grid with a small blend, must merge; where
        # the centre weights differ from node to node they cannot
        uniform = np.ptp(mx) == 0 and np.ptp(my) == 0 and not (wx or wy)
        assert merge or not (uniform and beta <= 0.5), beta
        assert not merge or uniform or beta == 0, beta
