"""Density and velocity of single cells against exact sums (math.fsum) of their
stored populations, over states whose populations span many binades, cancel,
vanish, or are too large for the float32 grids."""
import math

import numpy as np
import pytest

from oracle.lattice import velocities, weights
from tests.helpers import gpu

pytestmark = pytest.mark.gpu


def states(Q, rng):
    """(512 cells, Q) float32-representable fluctuations, a kind of state per 64 cells."""
    g = rng.standard_normal((512, Q))
    g[0:64] *= 0.01
    g[64:128] *= 10.0 ** rng.uniform(-12, 0, (64, Q))          # wide range within a cell
    g[128:192] *= 10.0 ** rng.uniform(-36, -24, (64, 1))       # all tiny
    g[192:256, 1::2] = -g[192:256, 2::2]                       # cancelling neighbours
    g[256:320] = 0.0                                           # rest, and a single value
    g[288:320, 5] = rng.standard_normal(32)
    g[320:384] = np.ldexp(1.0, rng.integers(-30, 3, (64, Q)))  # powers of two
    g[384:448] *= 1e-3
    g[384:448, 0] = 3.0                                        # one large value
    g[448:512] *= 1e33                                         # beyond the grids
    return g.astype(np.float32)


@pytest.mark.parametrize("model,storage", [("d3q19", "f32"), ("d3q27", "f32"), ("d3q19", "f16"), ("d3q27", "f16"),
                                           ("d3q27", "f64")])
def test_moments_of_single_cells_are_float64_sums(model, storage):
    lbm = gpu()
    Q = 19 if model == "d3q19" else 27
    w, e = weights(Q).numpy(), velocities(Q).numpy()
    g = states(Q, np.random.default_rng(9)).astype(np.float64)
    if storage == "f16":
        h = np.clip(g / w, -6e4, 6e4).astype(np.float16)
        raw = h
        g = (h.astype(np.float32) * w.astype(np.float32)).astype(np.float64)
    else:
        raw = g.astype({"f32": np.float32, "f64": np.float64}[storage])
    ctx = lbm.lbm_create(model, storage, (1, 1, 1), True, [], 1.7, 0.0)
    lbm.lbm_set_raw_state(ctx, 0, np.ascontiguousarray(raw.T).reshape(-1).view(np.uint8))
    lbm.lbm_stats_reset(ctx)
    lbm.lbm_stats_accumulate(ctx)
    rho, u = lbm.lbm_macroscopic(ctx, 0)
    mean, var, _ = lbm.lbm_stats_get(ctx, 0)
    assert np.array_equal(mean[0], rho) and np.array_equal(mean[1:], u)
    rho, u = rho.reshape(-1), u.reshape(3, -1)
    eps = 2.0 ** -53
    for c in range(512):
        size = math.fsum(abs(v) for v in g[c])
        want = 1.0 + math.fsum(g[c])
        # a float64 sum of Q terms is off by up to (Q - 1) eps sum |g|; 1 + adds one rounding
        assert abs(rho[c] - want) <= Q * eps * size + 2 * eps * abs(want), c
        for a in range(3):
            j = math.fsum(g[c] * e[:, a])
            if model == "d3q27":
                got, dj = u[a, c] * rho[c], Q * eps * size + 4 * eps * abs(j)
            else:
                got, dj = u[a, c], Q * eps * size + 2 * eps * abs(j)
            assert abs(got - j) <= dj, (c, a)
    # NaN and infinity stay what they are
    bad = raw.copy()
    bad[7, 3], bad[8, 4] = np.nan, np.inf
    lbm.lbm_set_raw_state(ctx, 0, np.ascontiguousarray(bad.T).reshape(-1).view(np.uint8))
    r2, u2 = lbm.lbm_macroscopic(ctx, 0)
    r2 = r2.reshape(-1)
    assert math.isnan(r2[7]) and r2[8] == np.inf
    keep = np.ones(512, bool)
    keep[7:9] = False
    assert np.array_equal(r2[keep], rho[keep])
    lbm.lbm_destroy(ctx)


@pytest.mark.parametrize("storage", ["f32", "f64"])
def test_velocity_of_diverged_cells_is_the_quotient(storage):
    """u = j / rho of cells whose density or momentum is infinite or whose density is zero."""
    lbm = gpu()
    e = velocities(27).numpy()
    px, mx = (int(np.flatnonzero((e == v).all(1))[0]) for v in ([1, 0, 0], [-1, 0, 0]))
    raw = np.zeros((512, 27), dtype={"f32": np.float32, "f64": np.float64}[storage])
    raw[:, px], raw[:, mx] = 0.5, -0.5              # j = (1, 0, 0)
    raw[0, 0], raw[1, 0] = np.inf, -np.inf          # rho infinite
    raw[2, 0] = -1.0                                # rho = 0
    raw[3, px] = np.inf                             # rho and j_x infinite
    ctx = lbm.lbm_create("d3q27", storage, (1, 1, 1), True, [], 1.7, 0.0)
    lbm.lbm_set_raw_state(ctx, 0, np.ascontiguousarray(raw.T).reshape(-1).view(np.uint8))
    lbm.lbm_stats_reset(ctx)
    lbm.lbm_stats_accumulate(ctx)
    g = raw.astype(np.float64)
    with np.errstate(all="ignore"):
        rho = 1.0 + g.sum(1)
        want = np.stack([g[:, e[:, a] > 0].sum(1) - g[:, e[:, a] < 0].sum(1) for a in range(3)]) / rho
    got_rho, got = lbm.lbm_macroscopic(ctx, 0)
    mean, _, _ = lbm.lbm_stats_get(ctx, 0)
    assert np.array_equal(got_rho.reshape(-1), rho)
    assert np.array_equal(got.reshape(3, -1), want, equal_nan=True)
    assert np.array_equal(mean[1:].reshape(3, -1), want, equal_nan=True)
    lbm.lbm_destroy(ctx)
