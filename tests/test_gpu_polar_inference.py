"""LearnableBiquadChain whose parameters are inference tensors (made, or
computed by a parametrization, under torch.inference_mode(); they keep no
version): it filters inside and outside that mode and gives the signal's
gradient, as with ordinary parameters."""
import pytest

from paper_2504_08624_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _setup():
    from paper_2504_08624_gb300 import api
    p = W.differentiable_chain_params(41, 2, 33)

    def make():
        return api.LearnableBiquadChain(p["rho"], p["phi"], p["b"], p["h"]).cuda()

    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    x = torch.randn(3, 5003, device="cuda", generator=g)
    m = make()
    with torch.no_grad():  # (no backward follows, so no plan is held for one)
        m(x)  # later calls run on this plan, whose tables the device then forms
        return make, m, x, m(x)


def test_made_in_inference_mode():
    make, m, x, want = _setup()
    with torch.inference_mode():
        layer = make()
        assert torch.equal(layer(x), want)
    with torch.no_grad():
        assert torch.equal(layer(x), want)
    grads = []
    for k in (layer, m):
        xi = x.clone().requires_grad_(True)
        grads += torch.autograd.grad(k(xi).square().sum(), [xi])
    assert torch.equal(*grads)


def test_computed_in_inference_mode():
    make, m, x, want = _setup()

    class Same(torch.nn.Module):
        def forward(self, v):
            return v * 1.0

    layer = make()
    torch.nn.utils.parametrize.register_parametrization(layer, "rho", Same())
    with torch.inference_mode():
        assert torch.equal(layer(x), want)
