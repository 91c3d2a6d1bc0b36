"""Device memory of a handle (host-side, no GPU): the scratch fields that its
kernels use and no others."""
import ctypes

import pytest

import inputs as I


@pytest.fixture(scope="module")
def B():
    import paper_1911_12913_gb300.binding as binding
    binding.load()
    return binding


def _bytes(B, walls, n=200, **kw):
    ax = I.wall_axis(n - 1, 0.0, 1.0) if walls else I.periodic_axis(n, 0.0, 1.0)
    grid, keep = B.make_grid(ax, ax)
    o = B.Opts()
    B.load().fdlbm_default_opts(ctypes.byref(o))
    for k, v in kw.items():
        setattr(o, k, v)
    return B.load().fdlbm_workspace_bytes(ctypes.byref(grid), ctypes.byref(o))


@pytest.mark.parametrize("walls", [False, True])
def test_scratch_fields(B, walls):
    n = 200
    field64 = 9 * 224 * n * 8  # rows of 224: 200 rounded up to 32
    tables = 16 * (n + n) * 8
    sweep = _bytes(B, walls, path=B.PATH_FUSED, rows_per_cta=4)  # a sweep: no scratch
    split = sweep + (2 if walls else 1) * field64 + tables
    assert _bytes(B, walls) == split
    assert _bytes(B, walls, path=B.PATH_STAGED) == split
    assert _bytes(B, walls, path=B.PATH_STAGED, scheme=B.SCHEME_T2S2_2) == sweep + 3 * field64
    f32 = _bytes(B, walls, precision=B.FP32_DEV)
    assert _bytes(B, walls, precision=B.FP32_DEV, path=B.PATH_STAGED) == f32 + 3 * field64 // 2
    if not walls:  # the adjoint takes its buffers from the caller
        assert _bytes(B, walls, adjoint=1) == split
        assert _bytes(B, walls, adjoint=1, path=B.PATH_FUSED, rows_per_cta=4) == sweep
        assert _bytes(B, walls, adjoint=1, precision=B.FP32_DEV) == f32


def test_batch_cases_keep_the_staged_kernels_scratch(B):
    ax = I.periodic_axis(200, 0.0, 1.0)
    grid, keep = B.make_grid(ax, ax)
    L = B.load()
    for precision, size in ((B.FP64, 8), (B.FP32_DEV, 4)):
        o = B.Opts()
        L.fdlbm_default_opts(ctypes.byref(o))
        o.precision = precision
        got = L.fdlbm_batch_workspace_bytes(1, ctypes.byref(grid), ctypes.byref(o))
        sweep = _bytes(B, False, precision=precision, path=B.PATH_FUSED, rows_per_cta=4)
        assert got == (sweep + 3 * 9 * 224 * 200 * size + 255) // 256 * 256
