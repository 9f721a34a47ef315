"""The action term's gradient on a stand-in system (marshalling only, no GPU): every segment
length gives the same, lengths below one are refused by the backward."""
import pytest
import torch

from paper_1705_02180_gb300 import autograd


class Quartic:
    """U = sum x^4 per frame: grad U = 4 x^3, H v = 12 x^2 v."""

    def energy_forces(self, topo, X, U, F=None):
        U.copy_((X.double() ** 4).sum((1, 2)))
        if F is not None:
            F.copy_(-4.0 * X ** 3)

    def hvp(self, topo, X, V, HV):
        HV.copy_(12.0 * X ** 2 * V)


def frames():
    return torch.randn(7, 5, 3, generator=torch.Generator().manual_seed(1)).requires_grad_()


@pytest.mark.parametrize("segment", [1, 3, 50])
def test_gradient_for_every_segment_length(segment):
    X = frames()
    w = torch.tensor(0.5, dtype=torch.float64, requires_grad=True)
    (G,) = torch.autograd.grad(w * autograd.force_norm_action(Quartic(), X, segment=segment), X,
                               create_graph=True)
    ref = (12.0 * X ** 2 * 8.0 * X ** 3).detach()
    assert torch.allclose(G.detach(), 0.5 * ref, rtol=1e-6)
    (gw,) = torch.autograd.grad(G.double().sum(), w)  # the incoming gradient stays differentiable
    assert torch.allclose(gw, ref.double().sum(), rtol=1e-6)


@pytest.mark.parametrize("segment", [0, -4])
def test_segments_below_one_are_refused_in_the_backward(segment):
    A = autograd.force_norm_action(Quartic(), frames(), segment=segment)
    assert A.item() > 0.0
    with pytest.raises((ValueError, RuntimeError)):
        A.backward()
