"""The input checks of long arrays that kernels do not read in place (registered
memory, odd addresses): refused wherever the bad value lies, and checked on the
device, not value by value on a host core."""
import ctypes
import time

import numpy as np
import pytest
import torch

from tests.helpers import gpu

pytestmark = pytest.mark.gpu

P = ctypes.POINTER(ctypes.c_double)
PIECE = 8 << 20   # values per staged piece


def array(n, place):
    """(float64 array of n values, what keeps its memory)."""
    if place == "ordinary":
        return np.empty(n), None
    if place == "odd":
        raw = np.empty(8 * n + 4, dtype=np.uint8)
        return raw[4:].view(np.float64), raw
    t = torch.empty(n, dtype=torch.float64).pin_memory()
    return t.numpy(), t


# 9 x 9 x 8 blocks: 27 populations are 1.07 pieces; density alone 0.04
@pytest.mark.parametrize("place", ["registered", "odd"])
def test_bad_values_are_found_in_every_piece(place):
    lbm = gpu()
    lib = lbm.load()
    ctx = lbm.lbm_create("d3q27", "f32", (9, 9, 8), True, [], 1.7, 0.0)
    n = ctx.ncells(0)
    assert PIECE < 27 * n < 2 * PIECE
    f, keep = array(27 * n, place)
    f[:] = 1.0 / 27
    f[5] = np.nan                                         # allowed: the cell is kept as it is
    call = lambda: lib.lbm_set_state(ctx.h, 0, ctypes.cast(f.ctypes.data, P), f.size)
    assert call() == lbm.LBM_OK
    before = lbm.lbm_get_raw_state(ctx, 0)
    for at in (0, PIECE - 1, PIECE, 27 * n - 1):
        for bad in (np.inf, -np.inf):
            old, f[at] = f[at], bad
            assert call() == lbm.LBM_ERR_NONFINITE, at
            f[at] = old
    rho, keep2 = array(n, place)
    u, keep3 = array(3 * n, place)
    rho[:], u[:] = 1.0, 0.0
    call = lambda: lib.lbm_init_equilibrium(ctx.h, 0, ctypes.cast(rho.ctypes.data, P), ctypes.cast(u.ctypes.data, P))
    for a, at, bad, status in ((rho, 0, 0.0, lbm.LBM_ERR_ARG), (rho, n - 1, -1.0, lbm.LBM_ERR_ARG),
                               (rho, n - 1, np.nan, lbm.LBM_ERR_NONFINITE), (u, 0, np.inf, lbm.LBM_ERR_NONFINITE),
                               (u, 3 * n - 1, np.nan, lbm.LBM_ERR_NONFINITE)):
        old, a[at] = a[at], bad
        assert call() == status, (at, bad)
        a[at] = old
    assert np.array_equal(lbm.lbm_get_raw_state(ctx, 0), before)
    assert call() == lbm.LBM_OK
    lbm.lbm_destroy(ctx)


def test_registered_arrays_cost_no_host_pass():
    """Density and velocity of 192^3 cells (28 M values).  One pass of a host
    core over them alone is longer than the whole call from ordinary memory;
    the copies of registered memory are not: each value crosses twice."""
    lbm = gpu()
    lib = lbm.load()
    ctx = lbm.lbm_create("d3q27", "f32", (24, 24, 24), True, [], 1.7, 0.0)
    n = ctx.ncells(0)
    best = {}
    for place in ("ordinary", "registered"):
        rho, keep = array(n, place)
        u, keep2 = array(3 * n, place)
        rho[:], u[:] = 1.0, 0.01
        times = []
        for _ in range(5):
            t = time.perf_counter()
            lbm._check(ctx, lib.lbm_init_equilibrium(ctx.h, 0, ctypes.cast(rho.ctypes.data, P),
                                                     ctypes.cast(u.ctypes.data, P)))
            times.append(time.perf_counter() - t)
        best[place] = min(times)
    lbm.lbm_destroy(ctx)
    print("\ninit of 192^3: ms", {k: round(1e3 * v, 2) for k, v in best.items()})
    assert best["registered"] <= 3 * best["ordinary"]
