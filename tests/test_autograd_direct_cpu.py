"""The direct first-order backward beside the differentiable node, on the CPU:
the kernels are stood in for by a linear map Y = x W, dx = g W^T, so that what
reaches them (and what is refused on the way) can be told."""

import pytest
import torch
import torch.autograd.forward_ad as fwad

from paper_2302_08381_gb300 import api, autograd

W = torch.arange(12.0, dtype=torch.float64).reshape(3, 4) - 5.0


@pytest.fixture
def y_of(monkeypatch):
    monkeypatch.setattr(api, "spherical_harmonics", lambda x, l_max, normalized: x.detach() @ W)
    monkeypatch.setattr(api, "backward", lambda x, g, l_max, normalized: g.detach() @ W.T)
    monkeypatch.setattr(api, "double_backward", lambda x, g, v, l_max, normalized, need_g=True, need_xyz=True: (
        v.detach() @ W if need_g else None, torch.zeros_like(x) if need_xyz else None))
    x = torch.randn(5, 3, dtype=torch.float64, requires_grad=True)
    return x, autograd.spherical_harmonics_autograd(x, 1)


def test_direct_and_differentiable_backward_agree(y_of):
    x, y = y_of
    g = torch.randn(5, 4, dtype=torch.float64, requires_grad=True)
    (d,) = torch.autograd.grad(y, x, g, retain_graph=True)
    (n,) = torch.autograd.grad(y, x, g, retain_graph=True, create_graph=True)
    assert not d.requires_grad and n.requires_grad
    assert torch.equal(d, n) and torch.equal(d, (g @ W.T).detach())
    (gg,) = torch.autograd.grad(n.sum(), g)
    assert torch.equal(gg, torch.ones(5, 3, dtype=torch.float64) @ W)


def test_broadcast_upstream_gradient(y_of):
    x, y = y_of
    y.sum().backward()  # its gradient is one expanded number
    assert torch.equal(x.grad, torch.ones(5, 4, dtype=torch.float64) @ W.T)


def test_forward_mode_over_the_backward_is_refused(y_of):
    """The backward has no forward-mode derivative: a tangent on the upstream
    gradient must raise, not be dropped."""
    x, y = y_of
    with fwad.dual_level():
        g = fwad.make_dual(torch.ones_like(y), torch.ones_like(y))
        with pytest.raises(NotImplementedError):
            torch.autograd.grad(y, x, g)


def test_batched_upstream_gradients_are_refused(y_of, monkeypatch):
    """is_grads_batched passes a gradient without storage of its own: its
    address, which the kernels take, must not be given out."""
    x, y = y_of
    monkeypatch.setattr(api, "backward", lambda x, g, l_max, normalized: g.contiguous().data_ptr())
    with pytest.raises(RuntimeError):
        torch.autograd.grad(y, x, torch.ones(2, 5, 4, dtype=torch.float64), is_grads_batched=True)
