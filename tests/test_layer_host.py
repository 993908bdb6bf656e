"""The autograd layer's outputs as a program uses them, with stand-ins for the
two library calls (y = 2 x, grad_x = 2 grad_y), so that no GPU is needed."""
import pytest
import torch

from paper_2607_20652_gb300 import dpb
from paper_2607_20652_gb300.layer import DPBLayer


@pytest.fixture
def layer(monkeypatch):
    def forward(plan, x, mu=None, sigma=None, workspace=None, stream=None, r_out=None, y=None):
        y = torch.empty_like(x) if y is None else y
        y.copy_(2 * x)
        code = torch.zeros((len(x), plan.code_len))
        return code.int(), code, x.norm(dim=1), y

    def backward(plan, x, idx, val, grad_y, sigma=None, workspace=None, stream=None, r=None):
        return 2 * grad_y, torch.zeros_like(val)

    monkeypatch.setattr(dpb, "forward", forward)
    monkeypatch.setattr(dpb, "backward", backward)
    monkeypatch.setattr(DPBLayer, "_stream", lambda self, device: None)
    return DPBLayer(d=64, levels=3, m_bits=12, children=16, beam=4, k=8, dtype="f32")


@pytest.mark.parametrize("shape", [(64,), (3, 64), (0, 64), (2, 3, 64), (2, 0, 64)])
def test_the_output_takes_in_place_work(layer, shape):
    x = torch.randn(shape, requires_grad=True)
    w = torch.randn(shape, requires_grad=True)
    y = layer(x)
    assert y.shape == x.shape and y.is_contiguous() and not y._is_view()
    y += w                          # a residual added in place
    torch.relu_(y)
    y.sum().backward()
    on = (2 * x.detach() + w.detach() > 0).float()
    assert torch.equal(x.grad, 2 * on) and torch.equal(w.grad, on)
    # without a gradient to the input, and under no_grad
    h = layer(x.detach())
    h += w
    assert torch.equal(torch.autograd.grad(h.sum(), w)[0], torch.ones_like(w))
    h = layer(x)
    with torch.no_grad():
        h *= 3.0
    assert torch.equal(torch.autograd.grad(h.sum(), x)[0], torch.full_like(x, 2.0))


def test_strided_input_and_expanded_gradient(layer):
    x = torch.randn(64, 4, 3).permute(2, 1, 0).requires_grad_(True)   # [3, 4, 64], not contiguous
    y = layer(x)
    assert torch.equal(y, 2 * x) and y.is_contiguous()
    y.sum().backward()                                                 # an expanded gradient
    assert torch.equal(x.grad, torch.full_like(x, 2.0))
