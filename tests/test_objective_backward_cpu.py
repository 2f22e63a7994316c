"""The objective's first-order backward refuses what its autograd function refuses (host only: a
handle that computes x . x on the CPU)."""
import pytest
import torch
from torch.autograd import forward_ad

from paper_2510_03932_gb300 import autograd


class Squares:
    def eval_obj(self, x):
        return (x.detach() * x.detach()).sum().reshape(1)

    def eval_grad_scaled(self, x, s):
        return 2.0 * x.detach() * s.detach()


def test_a_cotangent_with_a_tangent_is_refused():
    x = torch.arange(1.0, 4.0, dtype=torch.float64, requires_grad=True)
    F = autograd.objective(Squares(), x)
    one = torch.ones((), dtype=torch.float64)
    (g,) = torch.autograd.grad(F, x, one, retain_graph=True)
    assert torch.equal(g, 2.0 * x.detach())
    with forward_ad.dual_level():
        (g,) = torch.autograd.grad(F, x, one, retain_graph=True)   # a plain cotangent inside a level
        assert torch.equal(g, 2.0 * x.detach())
        with pytest.raises(NotImplementedError):
            torch.autograd.grad(F, x, forward_ad.make_dual(one, one))
