"""What the autograd function hands to the C entry points for tensors that are
taken in place: the values that the tensor stands for, read back here from the
memory that the library would read."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1206_0389_gb300 import autograd

N = 8


class FakeContext:
    Q = 27

    def dims(self, level):
        return (N, N, N)

    def ncells(self, level):
        return N ** 3


@pytest.fixture
def calls(monkeypatch):
    """Calls of the library, with the values behind each pointer."""
    seen = []

    def call(fn, ctx, *args):
        tensors = [a for a in args if torch.is_tensor(a)]
        seen.append((fn, [np.array(np.ctypeslib.as_array(
            ctypes.cast(t.data_ptr(), ctypes.POINTER(ctypes.c_double)), (t.numel(),))) for t in tensors]))
        for t in tensors:
            if fn in ("lbm_get_state", "lbm_adjoint_backward") and t is tensors[-1]:
                t.fill_(1.0)

    monkeypatch.setattr(autograd, "_in_place", lambda t: True)
    monkeypatch.setattr(autograd, "_call", call)
    monkeypatch.setattr(autograd.lbm, "lbm_set_state", lambda ctx, l, f: seen.append(("lbm_set_state", [])))
    monkeypatch.setattr(autograd.lbm, "lbm_adjoint_forward", lambda ctx, T, every: None)
    monkeypatch.setattr(autograd.lbm, "lbm_adjoint_generation", lambda ctx: (1, 1))
    return seen


def forms(x):
    """The same values as tensors of several kinds."""
    return {
        "plain": x.clone(),
        "pending sign": torch._neg_view(-x),
        "float32": x.float(),
        "pending sign, float32": torch._neg_view(-x.float()),
        "strided": torch.stack([x, x], -1)[..., 0],
        "imaginary part of a conjugate": torch.complex(x, -x).conj().imag,
        "expanded": x,
    }


@pytest.mark.parametrize("form", list(forms(torch.zeros(1))))
def test_force_and_gradient_reach_the_library_by_value(form, calls):
    g = torch.Generator().manual_seed(1)
    x = torch.randn(3, N, N, N, generator=g, dtype=torch.float32).double()
    lam = torch.randn(27, N, N, N, generator=g, dtype=torch.float32).double()
    if form == "expanded":
        x, lam = x[:, :1].expand(3, N, N, N), lam[:, :1].expand(27, N, N, N)
    F = forms(x)[form].detach().requires_grad_(True)
    fT = autograd.forced_fclb(F, FakeContext(), np.zeros((27, N, N, N)), 2, 1)
    fT.backward(forms(lam.to(F.dtype))[form].to(fT.dtype))
    by_name = dict(calls)
    assert np.array_equal(by_name["lbm_set_force"][0], x.reshape(-1).numpy())
    assert np.array_equal(by_name["lbm_adjoint_backward"][0], lam.reshape(-1).numpy())


def test_short_force_is_refused_before_the_context_changes(calls):
    F = torch.zeros(3, N, N, N - 1, dtype=torch.float64, requires_grad=True)
    with pytest.raises(ValueError):
        autograd.forced_fclb(F, FakeContext(), np.zeros((27, N, N, N)), 2, 1)
    assert calls == []
