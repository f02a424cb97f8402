"""LearnableBiquadChain with a parameter that holds its values lazily negated
(the imaginary part of a conjugate: one value of it is contiguous, and its
memory holds the opposite sign) filters as with the same values stored."""
import pytest

from paper_2504_08624_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["rho", "phi", "b", "h"])
def test_negated_view(name):
    from paper_2504_08624_gb300 import api
    p = W.differentiable_chain_params(41, 1, 33)
    m, want = (api.LearnableBiquadChain(p["rho"], p["phi"], p["b"], p["h"]).cuda() for _ in range(2))
    v = getattr(m, name).detach()
    if v.numel() == 1:
        z = torch.complex(torch.zeros_like(v), -v).conj().imag
    else:
        z = torch._neg_view(-v)
    assert z.is_neg() and z.is_contiguous() and torch.equal(z, v)
    setattr(m, name, torch.nn.Parameter(z))
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    x = torch.randn(2, 6001, device="cuda", generator=g)
    want(x)  # both then run on a reused plan, whose tables the device formed
    a, b = m(x), want(x)
    assert torch.max(torch.abs(a - b)) <= 1e-6 * torch.max(torch.abs(b))
    ga, gb = (torch.autograd.grad(y.square().mean(), list(k.parameters())) for y, k in ((a, m), (b, want)))
    for u, w in zip(ga, gb):
        assert torch.max(torch.abs(u - w)) <= 1e-6 * torch.max(torch.abs(w))
