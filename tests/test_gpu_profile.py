"""Launch counts and kinds of the timed launches (lbm_get_profile): one entry per
launch, the inflow, outlet and link launches under their own kind also where
coarse-to-fine work goes before them."""
import numpy as np
import pytest

from tests.helpers import gpu
from tests.test_gpu_graphs import make
from tests.test_gpu_nozzle import INFLOW, NOZ, NOZ1, nested_grid

pytestmark = pytest.mark.gpu

UPDATE, C2F, F2C, BC, OTHER = range(5)


# per coarse step of a 2-level grid: two substeps of the fine level, each with a
# coarse-to-fine launch, one restriction, one update of both levels and one of
# the fine level.  Nested FP16 grids update level 0 (near blocks, the rest) and
# set its ghosts in launches of their own.
@pytest.mark.parametrize("model", ["d3q19", "d3q27"])
@pytest.mark.parametrize("grid,storage,expect", [
    ("periodic", "f32", (1, 0, 0, 0, 0)),
    ("open", "f32", (1, 0, 0, 1, 0)),
    ("nozzle", "f16", (1, 0, 0, 2, 0)),
    # the refined cylinder meets the inflow: ghosts of both levels, then of the fine one
    ("nested", "f32", (2, 2, 1, 2, 0)),
    ("nested", "f16", (4, 2, 1, 3, 0)),
    # a nozzle inside the refined part: links with each substep of its level
    ("nested nozzle", "f32", (2, 2, 1, 3, 0)),
    # (every level-0 block touches the refined ones: no rest)
    ("nested nozzle", "f16", (3, 2, 1, 3, 0)),
])
def test_counts_per_kind(model, grid, storage, expect):
    lbm = gpu()
    if grid == "nozzle":
        ctx = lbm.lbm_create(model, storage, (5, 5, 5), False, [], 1.7, 0.18, nozzle=NOZ)
        lbm.lbm_set_inflow(ctx, *INFLOW)
    elif grid == "nested nozzle":
        nb, ref = nested_grid()
        ctx = lbm.lbm_create(model, storage, nb, False, ref, 1.7, 0.18, nozzle=NOZ1)
        lbm.lbm_set_inflow(ctx, *INFLOW)
    else:
        ctx = make(lbm, grid, model, storage)
    lbm.lbm_set_profiling(ctx, True)
    lbm.lbm_step(ctx, 3)
    ms, n = lbm.lbm_get_profile(ctx)
    lbm.lbm_destroy(ctx)
    assert tuple(n) == tuple(3 * k for k in expect)
    assert all((t > 0) == (k > 0) for t, k in zip(ms, n))
