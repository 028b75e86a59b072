"""Dense arrays of one call in different memories: registered, ordinary and
device ones side by side, and device arrays off an 8-byte boundary, in each of
the calls that take device arrays; the same values as with ordinary arrays."""
import ctypes

import numpy as np
import pytest
import torch

from tests.helpers import gpu

pytestmark = pytest.mark.gpu

P = ctypes.POINTER(ctypes.c_double)
PLACES = ["ordinary", "registered", "device", "device, odd address"]


class Array:
    """n float64 in a place, with the values of a NumPy array in and out."""

    def __init__(self, n, place, values=None):
        self.n, self.place = n, place
        if place == "ordinary":
            self.bytes = torch.zeros(8 * n, dtype=torch.uint8)
        elif place == "registered":
            self.bytes = torch.zeros(8 * n, dtype=torch.uint8).pin_memory()
        else:
            self.base = torch.zeros(8 * n + 8, dtype=torch.uint8, device="cuda")
            self.bytes = self.base[4:4 + 8 * n] if "odd" in place else self.base[:8 * n]
        if values is not None:
            self.bytes.copy_(torch.from_numpy(np.ascontiguousarray(values).reshape(-1).view(np.uint8)))
        torch.cuda.synchronize()
        self.ptr = ctypes.cast(self.bytes.data_ptr(), P)

    def get(self):
        return self.bytes.cpu().numpy().view(np.float64).copy()


def fields(ctx):
    rng = np.random.default_rng(3)
    n = ctx.ncells(0)
    return 1.0 + 0.02 * rng.standard_normal(n), 0.05 * rng.standard_normal(3 * n)


# 36 blocks: 18,432 values, checked on the host; 170: 87,040, on the device
@pytest.mark.parametrize("nb", [(3, 4, 3), (17, 2, 5)])
@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("p1", PLACES[:3])
@pytest.mark.parametrize("p2", PLACES[:3])
def test_density_and_velocity_apart(nb, storage, p1, p2):
    lbm = gpu()
    lib = lbm.load()
    got = []
    for a, b in (("ordinary", "ordinary"), (p1, p2)):
        ctx = lbm.lbm_create("d3q27", storage, nb, True, [], 1.7, 0.0)
        n = ctx.ncells(0)
        rho, u = fields(ctx)
        r, v = Array(n, a, rho), Array(3 * n, b, u)
        lbm._check(ctx, lib.lbm_init_equilibrium(ctx.h, 0, r.ptr, v.ptr))
        lbm.lbm_step(ctx, 3)
        ro, vo = Array(n, b), Array(3 * n, a)
        lbm._check(ctx, lib.lbm_macroscopic(ctx.h, 0, ro.ptr, vo.ptr))
        got.append(np.concatenate([ro.get(), vo.get()]))
        lbm.lbm_destroy(ctx)
    assert got[0].any() and np.array_equal(got[0], got[1])


@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("p1", PLACES)
@pytest.mark.parametrize("p2", PLACES)
def test_outputs_anywhere(storage, p1, p2):
    """Density and velocity, the state, and the gradient of an adjoint sweep."""
    lbm = gpu()
    lib = lbm.load()
    got = []
    for a, b in (("ordinary", "ordinary"), (p1, p2)):
        ctx = lbm.lbm_create("d3q27", storage, (2, 3, 2), True, [], 1.6, 0.0)
        n = ctx.ncells(0)
        rho, u = fields(ctx)
        lbm.lbm_init_equilibrium(ctx, 0, rho, u)
        lbm.lbm_set_force(ctx, 1e-3 * u)
        lbm.lbm_adjoint_forward(ctx, 4, 2)
        ro, vo, f, g = Array(n, a), Array(3 * n, b), Array(27 * n, a), Array(3 * n, b)
        lam = Array(27 * n, a.split(",")[0], np.tile(u, 9))
        lbm._check(ctx, lib.lbm_macroscopic(ctx.h, 0, ro.ptr, vo.ptr))
        lbm._check(ctx, lib.lbm_get_state(ctx.h, 0, f.ptr, f.n))
        lbm._check(ctx, lib.lbm_adjoint_backward(ctx.h, lam.ptr, g.ptr))
        got.append(np.concatenate([x.get() for x in (ro, vo, f, g)]))
        lbm.lbm_destroy(ctx)
    assert got[0].any() and np.array_equal(got[0], got[1])


def test_odd_device_inputs_are_refused():
    lbm = gpu()
    lib = lbm.load()
    ctx = lbm.lbm_create("d3q27", "f32", (2, 2, 2), True, [], 1.6, 0.0)
    rho, u = fields(ctx)
    v = Array(u.size, "device, odd address", u)
    assert lib.lbm_init_equilibrium(ctx.h, 0, None, v.ptr) == lbm.LBM_ERR_ARG
    lbm.lbm_destroy(ctx)
