"""Dense arrays between the caller and the block storage: the launch that
reads or writes ordinary memory in place against the slab-by-slab copies
(which registered memory takes), on short and long arrays, at odd starts; the
input checks on the device and on the host; device tensors in autograd."""
import ctypes

import numpy as np
import pytest
import torch

from tests.helpers import gpu

pytestmark = pytest.mark.gpu

P = ctypes.POINTER(ctypes.c_double)


def ordinary(n, start):
    """n float64 that start `start` elements into fresh, untouched memory."""
    return np.empty(n + start)[start:]


def ordinary_at_start(n, dtype=np.float64):
    return np.empty(n, dtype=dtype)


def registered(n, start):
    return torch.empty(n + start, dtype=torch.float64).pin_memory().numpy()[start:]


def ptr(a):
    return a.ctypes.data_as(P)


# the largest case: 20 MB per component (two touching threads), 27 components
@pytest.mark.parametrize("nb", [(1, 1, 1), (3, 2, 5), (18, 17, 16)])
@pytest.mark.parametrize("model,storage", [("d3q27", "f32"), ("d3q19", "f16"), ("d3q27", "f64")])
def test_in_place_transfers_equal_copies(nb, model, storage):
    lbm = gpu()
    lib = lbm.load()
    rng = np.random.default_rng(5)
    n = 512 * nb[0] * nb[1] * nb[2]
    got = []
    for make, start in ((registered, 0), (ordinary, 0), (ordinary, 3)):
        ctx = lbm.lbm_create(model, storage, nb, True, [], 1.7, 0.1)
        rng = np.random.default_rng(5)
        u = make(3 * n, start)
        u[:] = 0.05 * rng.standard_normal(3 * n)
        lbm._check(ctx, lib.lbm_init_equilibrium(ctx.h, 0, None, ptr(u)))     # rho filled
        rho = make(n, start)
        rho[:] = 1.0 + 0.02 * rng.standard_normal(n)
        f = make(ctx.Q * n, start)
        lbm._check(ctx, lib.lbm_get_state(ctx.h, 0, ptr(f), f.size))
        out = [f.copy()]
        lbm._check(ctx, lib.lbm_init_equilibrium(ctx.h, 0, ptr(rho), ptr(u)))
        f *= 1.001
        f[::1001] = np.nan                                                    # kept as they are
        lbm._check(ctx, lib.lbm_set_state(ctx.h, 0, ptr(f), f.size))
        if model == "d3q27" and storage != "f16":
            F = make(3 * n, start)
            F[:] = 1e-5 * rng.standard_normal(3 * n)
            lbm._check(ctx, lib.lbm_set_force(ctx.h, ptr(F)))
        r, v = make(n, start), make(3 * n, start)
        lbm._check(ctx, lib.lbm_macroscopic(ctx.h, 0, ptr(r), ptr(v)))
        lbm._check(ctx, lib.lbm_stats_reset(ctx.h))
        lbm._check(ctx, lib.lbm_stats_accumulate(ctx.h))
        m, s = make(4 * n, start), make(3 * n, start)
        lbm._check(ctx, lib.lbm_stats_get(ctx.h, 0, ptr(m), ptr(s), None))
        cells = np.array([0, n - 1, n // 2, -1, n], dtype=np.int64)
        c = make(5 * ctx.Q, start)
        lbm._check(ctx, lib.lbm_get_cells(ctx.h, 0, 5, cells.ctypes.data_as(ctypes.POINTER(ctypes.c_int64)), ptr(c)))
        got.append([a.copy() for a in out + [r, v, m, s, c]] + [lbm.lbm_get_raw_state(ctx, 0)])
        lbm.lbm_destroy(ctx)
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert np.array_equal(a, b, equal_nan=a.dtype.kind == "f")


@pytest.mark.parametrize("nb", [(1, 1, 1), (5, 4, 3)])      # checked on the host; long enough for the device
@pytest.mark.parametrize("offset", [1, 4])
def test_arrays_at_odd_addresses(nb, offset):
    """Buffer views that start off an 8-byte boundary take the copies."""
    lbm = gpu()
    lib = lbm.load()
    n = 512 * nb[0] * nb[1] * nb[2]

    def odd(size, dtype=np.float64):
        a = np.frombuffer(bytearray(8 * size + offset), dtype=dtype, offset=offset)
        assert a.ctypes.data % 8 == offset
        return a

    got = []
    for make in (ordinary_at_start, odd):
        rng = np.random.default_rng(7)
        ctx = lbm.lbm_create("d3q27", "f32", nb, True, [], 1.7, 0.0)
        rho, u, F = make(n), make(3 * n), make(3 * n)
        rho[:] = 1.0 + 0.02 * rng.standard_normal(n)
        u[:] = 0.05 * rng.standard_normal(3 * n)
        F[:] = 1e-5 * rng.standard_normal(3 * n)
        lbm._check(ctx, lib.lbm_init_equilibrium(ctx.h, 0, ptr(rho), ptr(u)))
        lbm._check(ctx, lib.lbm_set_force(ctx.h, ptr(F)))
        lbm.lbm_step(ctx, 2)
        f, r, v = make(27 * n), make(n), make(3 * n)
        lbm._check(ctx, lib.lbm_get_state(ctx.h, 0, ptr(f), f.size))
        lbm._check(ctx, lib.lbm_set_state(ctx.h, 0, ptr(f), f.size))
        lbm._check(ctx, lib.lbm_macroscopic(ctx.h, 0, ptr(r), ptr(v)))
        cells, c = make(n, np.int64), make(27 * n)
        cells[:] = rng.permutation(n)
        lbm._check(ctx, lib.lbm_get_cells(ctx.h, 0, n, cells.ctypes.data_as(ctypes.POINTER(ctypes.c_int64)), ptr(c)))
        lbm.lbm_adjoint_forward(ctx, 2, 0)
        g = make(3 * n)
        lbm._check(ctx, lib.lbm_adjoint_backward(ctx.h, ptr(f), ptr(g)))
        got.append([a.copy() for a in (f, r, v, c, g)])
        lbm.lbm_destroy(ctx)
    for a, b in zip(*got):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("make", [ordinary, registered])
@pytest.mark.parametrize("nb", [(1, 2, 1), (5, 4, 3)])      # checked on the host; on the device where within reach
def test_refused_arrays_change_nothing(make, nb):
    lbm = gpu()
    lib = lbm.load()
    n = 512 * nb[0] * nb[1] * nb[2]
    ctx = lbm.lbm_create("d3q27", "f32", nb, True, [], 1.7, 0.0)
    before = lbm.lbm_get_raw_state(ctx, 0)
    rho, u, f, F = make(n, 1), make(3 * n, 1), make(27 * n, 1), make(3 * n, 1)
    for a, v in ((rho, 1.0), (u, 0.01), (f, 0.1), (F, 0.0)):
        a[:] = v

    def status(call, a, at, bad):
        good = a[at]
        a[at] = bad
        st = call()
        a[at] = good
        return st

    init = lambda: lib.lbm_init_equilibrium(ctx.h, 0, ptr(rho), ptr(u))
    for at in (0, n - 1, -1):
        for bad in (np.nan, np.inf, -np.inf):
            assert status(init, rho, at, bad) == lbm.LBM_ERR_NONFINITE
            assert status(init, u, at, bad) == lbm.LBM_ERR_NONFINITE
            assert status(lambda: lib.lbm_set_force(ctx.h, ptr(F)), F, at, bad) == lbm.LBM_ERR_NONFINITE
        for bad in (0.0, -0.0, -1.0):
            assert status(init, rho, at, bad) == lbm.LBM_ERR_ARG
        for bad in (np.inf, -np.inf):
            assert status(lambda: lib.lbm_set_state(ctx.h, 0, ptr(f), f.size), f, at, bad) == lbm.LBM_ERR_NONFINITE
    assert np.array_equal(lbm.lbm_get_raw_state(ctx, 0), before)
    assert init() == lbm.LBM_OK
    lbm.lbm_destroy(ctx)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_autograd_on_the_gpu_equals_the_host(dtype):
    """F on the GPU (arrays in place, from a side stream) and on the host."""
    from paper_1206_0389_gb300.autograd import forced_fclb
    lbm = gpu()
    g = torch.Generator().manual_seed(3)
    F0 = (1e-4 * torch.randn((3, 16, 8, 24), generator=g, dtype=torch.float64)).to(dtype)
    f0 = torch.full((27, 16, 8, 24), 1.0 / 27, dtype=torch.float64) * (1 + 0.02 * torch.randn((27, 16, 8, 24), generator=g, dtype=torch.float64))
    w = torch.randn(f0.shape, generator=g, dtype=torch.float64).to(dtype)
    out = []
    for dev in ("cpu", "cuda"):
        ctx = lbm.lbm_create("d3q27", "f32", (3, 1, 2), True, [], 1.8, 0.0)
        with torch.cuda.stream(torch.cuda.Stream()):
            F = F0.to(dev).transpose(1, 3).contiguous().transpose(1, 3).requires_grad_(True)   # not contiguous
            fT = forced_fclb(F, ctx, f0.numpy(), 5, 0)
            (fT * w.to(dev)).sum().backward()
            out.append((fT.detach().cpu(), F.grad.cpu()))
        lbm.lbm_destroy(ctx)
    assert out[0][0].dtype == dtype and out[1][1].dtype == dtype
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
