"""Grids whose voxels 32-bit offsets cannot number are refused before any size is computed or any
device is touched (no GPU needed)."""
import ctypes as C

import pytest

from synth import workload_params


@pytest.fixture(scope="module")
def tg():
    from paper_1810_05370_gb300.build import build
    build()
    from paper_1810_05370_gb300 import _tg
    return _tg


REFUSED = [(2048, 1024, 1024), (1 << 20, 1 << 20, 1 << 20), (4, 1 << 20, 512), (2048, 2048, 2048)]
ACCEPTED = [(2047, 1024, 1024), (4, 1 << 20, 511), (1290, 1290, 1290)]


@pytest.mark.parametrize("n", REFUSED)
def test_refused(tg, n):
    grid, params = tg.make_grid(n), tg.make_params(workload_params())
    for prec in (tg.TG_FP64, tg.TG_MIXED):
        assert tg.tg_workspace_bytes(grid, None, prec) == 0
        assert tg.tg_workspace_bytes_adjoint(grid, params, prec) == 0
        state, ctx = tg.tg_state(), C.c_void_p()
        for q in ("p", "i", "n", "g", "w", "f", "o", "l", "bg"):
            setattr(state, q, 256)       # never read: the grid is refused first
        for a in range(3):
            state.u[a] = state.v[a] = 256
        rc = tg.lib.tg_init(C.byref(grid), C.byref(params), prec, C.byref(state), C.c_void_p(256),
                            C.c_size_t(1 << 62), None, 0, C.byref(ctx), None)
        assert rc == tg.TG_ERR_ARG and not ctx.value
    assert tg.tg_tape_bytes(grid) == 0


@pytest.mark.parametrize("n", ACCEPTED)
def test_accepted(tg, n):
    grid = tg.make_grid(n)
    voxels = n[0] * n[1] * n[2]
    for prec in (tg.TG_FP64, tg.TG_MIXED):
        assert tg.tg_workspace_bytes(grid, None, prec) > 8 * voxels
    assert tg.tg_tape_bytes(grid) >= 26 * 8 * voxels
