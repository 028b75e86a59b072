"""The inflow disc at its rim: which face cells carry the inflow is decided in
float64, behind a float32 test that only lets clearly outside cells go."""
import numpy as np
import pytest

from tests.helpers import gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("axis", [(12.0, 8.0), (11.5, 8.5), (0.1, 15.9), (-3.0, 20.0), (1.0e5, 8.0)])
@pytest.mark.parametrize("diameter", [0.0, 5.0, 6.0, 10.0, 2.0e5])
def test_disc_cells_at_the_rim(axis, diameter):
    """Radii through cell centres (3, 4, 5 triangles), a hair below and above."""
    lbm = gpu()
    NY, NZ = 24, 16
    y, z = np.arange(NY) + 0.5, np.arange(NZ)[:, None] + 0.5
    for scale in (1.0, 1.0 - 2.0 ** -50, 1.0 + 2.0 ** -50):
        D = diameter * scale
        ctx = lbm.lbm_create("d3q27", "f64", (2, 3, 2), False, [], 1.7, 0.0)
        lbm.lbm_set_inflow(ctx, axis[0], axis[1], D, 0.1, 0.0, 1)
        lbm.lbm_step(ctx, 1)
        _, u = lbm.lbm_macroscopic(ctx, 0)
        lbm.lbm_destroy(ctx)
        dy, dz = y - axis[0], z - axis[1]
        disc = dy * dy + dz * dz < (0.5 * D) * (0.5 * D)
        # cells whose whole 3 x 3 neighbourhood on the face agrees move like it
        near = [np.roll(disc, (a, b), (0, 1)) for a in (-1, 0, 1) for b in (-1, 0, 1)]
        every, none = np.all(near, 0), ~np.any(near, 0)
        assert (np.abs(u[0, :, :, 0][none]) == 0.0).all()
        full = u[0, :, :, 0][every]
        assert full.size == 0 or (full > 0.01).all() and np.ptp(full) < 1e-15
        # and a face cell's own straight population tells its rim apart
        f = np.abs(u[0, :, :, 0])
        assert (f[disc] > f[none].max(initial=0.0)).all()
