"""Host threads that drive contexts of their own, of one model and storage but
of sizes on both sides of the rule that cuts blocks into runs: the bits of the
same runs one after the other."""
import threading

import numpy as np
import pytest

from tests.helpers import gpu

pytestmark = pytest.mark.gpu

SIZES = [(1, 2, 3), (9, 8, 8), (4, 4, 4), (16, 12, 9)]


@pytest.mark.parametrize("model,storage", [("d3q27", "f32"), ("d3q19", "f16"), ("d3q27", "f64")])
def test_contexts_of_several_threads(model, storage, monkeypatch):
    lbm = gpu()
    monkeypatch.setenv("LBM_LAUNCH_SHAPE", "128,8,0")

    def run(k, out):
        ctx = lbm.lbm_create(model, storage, SIZES[k], True, [], 1.7, 0.1)
        NX, NY, NZ = ctx.dims(0)
        u = 0.03 * np.random.default_rng(k).standard_normal((3, NZ, NY, NX))
        lbm.lbm_init_equilibrium(ctx, 0, None, u)
        for n in (1, 16, 3, 33):
            lbm.lbm_step(ctx, n)
        out[k] = lbm.lbm_get_raw_state(ctx, 0)
        lbm.lbm_destroy(ctx)

    alone, together = {}, {}
    for k in range(len(SIZES)):
        run(k, alone)
    threads = [threading.Thread(target=run, args=(k, together)) for k in range(len(SIZES))]
    for t in threads:
        t.start()
    for t in threads:
        t.join(120)
    for k in range(len(SIZES)):
        assert alone[k].any() and np.array_equal(alone[k], together[k]), SIZES[k]
