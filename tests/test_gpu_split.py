"""Short work lists cut each block into runs of cells, one CTA per run; long
ones give a CTA the whole block.  A state that repeats along z evolves on a
long grid as on one period, so both sides of the rule meet bit for bit (one
launch shape: one compiled kernel)."""
import numpy as np
import pytest

from tests.helpers import gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model", ["d3q19", "d3q27"])
@pytest.mark.parametrize("storage", ["f64", "f32", "f16"])
@pytest.mark.parametrize("shape", ["128,1,0", "128,8,0", "256,4,0", "128,8,1"])
@pytest.mark.parametrize("walls", [0, 3])
def test_split_blocks_match_whole_blocks(model, storage, shape, walls, monkeypatch):
    """One period of 2 x 3 x 1 blocks (split fourfold) against 2 x 3 x n with
    n = 17 (102 blocks), 101 (606) and 304 (1824): split fourfold, in two, not
    at all, whatever the residency (2 to 8 CTAs on 152 SMs)."""
    lbm = gpu()
    monkeypatch.setenv("LBM_LAUNCH_SHAPE", shape)
    rng = np.random.default_rng(11)
    rho = 1.0 + 0.02 * rng.standard_normal((8, 24, 16))
    u = 0.03 * rng.standard_normal((3, 8, 24, 16))

    def run(n):
        ctx = lbm.lbm_create(model, storage, (2, 3, n), True, [], 1.7, 0.1, walls=walls)
        lbm.lbm_init_equilibrium(ctx, 0, np.tile(rho, (n, 1, 1)), np.tile(u, (1, n, 1, 1)))
        lbm.lbm_step(ctx, 3)
        raw = lbm.lbm_get_raw_state(ctx, 0).reshape(n, -1)
        lbm.lbm_destroy(ctx)
        return raw

    one = run(1)
    assert one.any()
    for n in (17, 101, 304):
        assert (run(n) == one).all(), n
