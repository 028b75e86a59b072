"""When runs of steps go out as graphs of 16: not before that pays, and with the
bits of single steps on every grid, from either parity, also after a change."""
import time

import numpy as np
import pytest

import synth
from tests.helpers import gpu
from tests.test_gpu_graphs import make, states

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", ["open", "nested", "three"])
@pytest.mark.parametrize("model,storage", [("d3q27", "f32"), ("d3q19", "f16"), ("d3q27", "f16"), ("d3q19", "f64")])
def test_long_runs_equal_single_steps(grid, model, storage, monkeypatch):
    """256 steps are past the threshold of every grid (at most 14 launches a
    step), the calls before and after cross it and flip the parity."""
    lbm = gpu()
    monkeypatch.setenv("LBM_LAUNCH_SHAPE", "128,8,0")
    out = []
    for single in (False, True):
        ctx = make(lbm, grid, model, storage)
        for n in (24, 25, 256, 17, 40):
            for k in ([1] * n if single else [n]):
                lbm.lbm_step(ctx, k)
            if n == 256:
                lbm.lbm_set_inflow(ctx, 4.0 * ctx.nb[1], 4.0 * ctx.nb[2], 12.0, 0.04, 0.2, 4)
        assert lbm.lbm_get_step(ctx) == 362
        out.append(states(lbm, ctx))
        lbm.lbm_destroy(ctx)
    for a, b in zip(*out):
        assert a.any() and np.array_equal(a, b)


@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_changing_the_inflow_every_16_steps_costs_no_long_capture(storage):
    """Three levels: 16 steps in one call after each change of the inflow take no
    longer than 16 calls of one step after such a change.  (Capturing 16 steps
    took half as long again; allowed: a fifth for the clock.)"""
    lbm = gpu()
    flags, (y0, z0) = synth.jet_three_level(16, 8, 8, r1=(0.0, 12.0), r2=(0.0, 8.0), x1=(0, 48), x2=(0, 24))
    ctx = lbm.lbm_create("d3q27", storage, (16, 8, 8), False, flags, 1.7, 0.0)
    took = {1: [], 16: []}
    for r in range(24):
        for n in took:
            lbm.lbm_set_inflow(ctx, y0, z0, 8.0, 0.05 - 1e-4 * (r % 2), 0.01, 3)
            lbm.lbm_sync(ctx)
            t = time.perf_counter()
            for _ in range(16 // n):
                lbm.lbm_step(ctx, n)
            lbm.lbm_sync(ctx)
            took[n].append(time.perf_counter() - t)
    lbm.lbm_destroy(ctx)
    one, many = (float(np.median(took[n][2:])) for n in (1, 16))
    print("\n16 steps after a change, us: calls of one %.0f, one call %.0f" % (1e6 * one, 1e6 * many))
    assert many <= 1.2 * one
