"""The adjoint step on ragged boxes (one block wide: every neighbour wraps) with
forces large enough that every term of the force counts, against the float64
oracle's autograd gradient."""
import numpy as np
import pytest
import torch

import synth
from oracle.adjoint import kinetic_energy_loss, reference_gradient
from oracle.collision import feq_fclb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [(1, 1, 1), (1, 2, 3)])
@pytest.mark.parametrize("sigma,zero", [(0.0, True), (1e-2, False)])
@pytest.mark.parametrize("every", [1, 2])
def test_gradient_on_ragged_boxes(nb, sigma, zero, every):
    from paper_1206_0389_gb300 import lbm
    from paper_1206_0389_gb300.autograd import forced_fclb
    NX, NY, NZ = (8 * n for n in nb)
    rng = np.random.default_rng(7)
    rho = torch.from_numpy(1.0 + 0.05 * rng.standard_normal(NX * NY * NZ))
    u = torch.from_numpy(0.05 * rng.standard_normal((3, NX * NY * NZ)))
    f0 = feq_fclb(rho, u).reshape(27, NZ, NY, NX)
    f0 = f0 * (1.0 + 0.05 * torch.from_numpy(rng.standard_normal(f0.shape)))
    F = sigma * rng.standard_normal((3, NZ, NY, NX))
    region = (0, NZ, 0, NY, 0, NX // 2)
    Lo, go = reference_gradient(f0, torch.from_numpy(F), nb, 1.3, 3, region)
    ctx = lbm.lbm_create("d3q27", "f64", nb, True, [], 1.3, 0.0)
    Ft = torch.from_numpy(F).clone().requires_grad_(True)
    fT = forced_fclb(Ft, ctx, f0.numpy(), 3, every)
    L = kinetic_energy_loss(fT, Ft, region)
    L.backward()
    lbm.lbm_destroy(ctx)
    # float64 against float64: the bound of the existing gradient test
    assert abs(float(L.detach()) - Lo) <= 1e-9 * abs(Lo)
    assert float((Ft.grad - go).abs().max()) <= 1e-10 * float(go.abs().max())
