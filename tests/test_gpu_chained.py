"""Chained launches against launches that never overlap: the same bits.  The
boxes are small, so that every CTA of a launch is resident and the next two
launches come up while it still runs."""
import os
import subprocess
import sys

import numpy as np
import pytest

from tests.helpers import gpu
from tests.test_gpu_graphs import make, states
from tests.test_gpu_nozzle import INFLOW, NOZ

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", ["periodic", "walls", "open", "tank", "nozzle"])
@pytest.mark.parametrize("model,storage", [("d3q19", "f32"), ("d3q27", "f32"), ("d3q19", "f16"), ("d3q27", "f16"),
                                           ("d3q19", "f64"), ("d3q27", "f64")])
@pytest.mark.parametrize("shape", ["128,8,0", "256,1,0"])
def test_graph_of_steps_equals_single_launches(grid, model, storage, shape, monkeypatch):
    """41 steps: two graphs of 16 and nine of one; the other side launches
    kernel after kernel with a host wait between (timed launches)."""
    lbm = gpu()
    monkeypatch.setenv("LBM_LAUNCH_SHAPE", shape)
    out = []
    for direct in (False, True):
        if grid == "tank":
            f = np.zeros((4, 4, 6), bool)
            f[1:3, 1:3, 1:4] = True
            ctx = lbm.lbm_create(model, storage, (6, 4, 4), False, [f], 1.8, 0.18, walls=15, slip=8, outlet=1)
            lbm.lbm_set_inflow(ctx, 16.0, 16.0, 9.0, 0.05, 0.2, 3)
        elif grid == "nozzle":
            ctx = lbm.lbm_create(model, storage, (5, 5, 5), False, [], 1.7, 0.18, nozzle=NOZ)
            lbm.lbm_set_inflow(ctx, *INFLOW)
        else:
            ctx = make(lbm, grid, model, storage)
        lbm.lbm_set_profiling(ctx, direct)
        lbm.lbm_step(ctx, 41)
        out.append(states(lbm, ctx))
        lbm.lbm_destroy(ctx)
    for a, b in zip(*out):
        assert a.any() and np.array_equal(a, b)


GRADIENT = """
import sys
import numpy as np
from paper_1206_0389_gb300 import lbm
out = {}
for nb in ((1, 1, 1), (1, 2, 3), (3, 3, 2)):
    for sigma in (0.0, 1e-2):
        rng = np.random.default_rng(7)
        ctx = lbm.lbm_create("d3q27", "f32", nb, True, [], 1.3, 0.0)
        NX, NY, NZ = ctx.dims(0)
        lbm.lbm_init_equilibrium(ctx, 0, 1 + 0.05 * rng.standard_normal((NZ, NY, NX)),
                                 0.05 * rng.standard_normal((3, NZ, NY, NX)))
        lbm.lbm_set_force(ctx, sigma * rng.standard_normal((3, NZ, NY, NX)))
        for every in (1, 5):
            lbm.lbm_adjoint_forward(ctx, 24, every)
            key = "%s_%g_%d" % (nb, sigma, every)
            out["f" + key] = lbm.lbm_get_state(ctx, 0)
            out["g" + key] = lbm.lbm_adjoint_backward(ctx, rng.standard_normal((27, NZ, NY, NX)))
        lbm.lbm_destroy(ctx)
np.savez(sys.argv[1], **out)
"""


def test_chained_gradient_equals_blocking_launches(tmp_path):
    """FP32 forward and reverse sweeps (both chained) in one process, and in
    another that waits for each launch on the host (CUDA_LAUNCH_BLOCKING)."""
    got = []
    for blocking in ("0", "1"):
        path = str(tmp_path / ("g%s.npz" % blocking))
        env = dict(os.environ, CUDA_LAUNCH_BLOCKING=blocking, LBM_LAUNCH_SHAPE="128,8,0")
        subprocess.run([sys.executable, "-c", GRADIENT, path], check=True, env=env, timeout=300,
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
        got.append(np.load(path))
    assert len(got[0].files) == 24
    for k in got[0].files:
        assert got[0][k].any() and np.array_equal(got[0][k], got[1][k]), k
