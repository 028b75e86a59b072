"""Runs of coarse steps that go out as one graph of many steps, against the
same steps one call at a time: the same bits, from either parity and around a
change of the inflow."""
import numpy as np
import pytest

import synth
from tests.helpers import gpu

pytestmark = pytest.mark.gpu


def make(lbm, grid, model, storage, stream=None):
    kw = {}
    if grid == "periodic":
        ctx = lbm.lbm_create(model, storage, (3, 1, 2), True, [], 1.7, 0.1, stream)
    elif grid == "walls":
        ctx = lbm.lbm_create(model, storage, (3, 2, 2), True, [], 1.7, 0.1, stream, walls=15, slip=8)
    elif grid == "open":
        ctx = lbm.lbm_create(model, storage, (4, 2, 2), False, [], 1.7, 0.1, stream, outlet=1)
    elif grid == "nested":
        f = np.zeros((5, 5, 6), bool)
        f[2, 2, :] = True
        ctx = lbm.lbm_create(model, storage, (6, 5, 5), False, [f], 1.8, 0.18, stream)
    else:
        flags, _ = synth.jet_three_level(6, 8, 8, r1=(0.0, 16.0), r2=(0.0, 8.0), x1=(0, 40), x2=(0, 24))
        ctx = lbm.lbm_create(model, storage, (6, 8, 8), False, flags, 1.8, 0.18, stream)
    rng = np.random.default_rng(2)
    for l in range(ctx.levels):
        NX, NY, NZ = ctx.dims(l)
        lbm.lbm_init_equilibrium(ctx, l, None, 0.02 * rng.standard_normal((3, NZ, NY, NX)))
    if grid not in ("periodic", "walls"):
        lbm.lbm_set_inflow(ctx, 4.0 * ctx.nb[1], 4.0 * ctx.nb[2], 10.0, 0.05, 0.2, 3)
    return ctx


def states(lbm, ctx):
    return [lbm.lbm_get_raw_state(ctx, l) for l in range(ctx.levels)]


@pytest.mark.parametrize("grid", ["periodic", "walls", "open", "nested", "three"])
@pytest.mark.parametrize("model,storage", [("d3q27", "f32"), ("d3q19", "f16"), ("d3q27", "f16")])
def test_many_steps_equal_single_steps(grid, model, storage, monkeypatch):
    lbm = gpu()
    monkeypatch.setenv("LBM_LAUNCH_SHAPE", "128,8,0")
    out = []
    for single in (False, True):
        ctx = make(lbm, grid, model, storage)
        for n in (16, 1, 37, 15, 32):
            for k in ([1] * n if single else [n]):
                lbm.lbm_step(ctx, k)
            if n == 37 and grid not in ("periodic", "walls"):
                lbm.lbm_set_inflow(ctx, 4.0 * ctx.nb[1], 4.0 * ctx.nb[2], 12.0, 0.04, 0.2, 4)
        assert lbm.lbm_get_step(ctx) == 101
        out.append(states(lbm, ctx))
        lbm.lbm_destroy(ctx)
    for a, b in zip(*out):
        assert np.array_equal(a, b)
