"""LearnableBiquadChain straight from its parameters (one launch for the
coefficients, one for their gradients) against the same module through
rows() by torch ops: the output is the same, every gradient agrees to 1e-12
of its largest value (FP64 chain rule on the same dL/d(rows)), parameters
may be frozen or changed in place before the backward, and create_graph gives
gradients that can be differentiated again."""
import pytest

from paper_2504_08624_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _models(n=4, taps=33, seed=41):
    from paper_2504_08624_gb300 import api

    class ByRows(api.LearnableBiquadChain):
        def rows(self):
            return super().rows()

    p = W.differentiable_chain_params(seed, n, taps)
    # a newly built plan takes its FIR's spectrum from the host's FP64
    # transform, a reused one from the device's: start from a reused one
    with torch.no_grad():
        api.LearnableBiquadChain(p["rho"], p["phi"], p["b"], p["h"]).cuda()(_signals()[0])
    return [c(p["rho"], p["phi"], p["b"], p["h"]).cuda() for c in (api.LearnableBiquadChain, ByRows)]


def _signals(C=3, Ns=9001):
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    return torch.randn(C, Ns, device="cuda", generator=g), torch.randn(C, Ns, device="cuda", generator=g)


@pytest.mark.parametrize("frozen", [(), ("rho",), ("b", "h"), ("rho", "phi", "b", "h")])
def test_gradients_as_by_rows(frozen):
    x, t = _signals()
    got = []
    for m in _models():
        for k in frozen:
            getattr(m, k).requires_grad_(False)
        xi = x.clone().requires_grad_(True)
        y = m(xi)
        from paper_2504_08624_gb300 import api
        api.mse_loss(y, t).backward()
        got.append((y.detach(), xi.grad, {k: p.grad for k, p in m.named_parameters()}))
    (y0, dx0, g0), (y1, dx1, g1) = got
    assert torch.equal(y0, y1) and torch.equal(dx0, dx1)
    for k in g0:
        assert (g0[k] is None) == (g1[k] is None) == (k in frozen)
        if g0[k] is not None:
            assert g0[k].shape == g1[k].shape
            assert torch.max(torch.abs(g0[k] - g1[k])) <= 1e-12 * torch.max(torch.abs(g1[k])), k


def test_parameters_changed_before_the_backward():
    x, t = _signals()
    got = []
    for m in _models():
        y = m(x)
        with torch.no_grad():
            for p in m.parameters():
                p.mul_(0.5)
        (y * t).sum().backward()
        got.append([p.grad for p in m.parameters()])
    for a, b in zip(*got):
        assert torch.max(torch.abs(a - b)) <= 1e-12 * torch.max(torch.abs(b))


def test_create_graph():
    x, t = _signals()
    got = []
    for m in _models():
        g = torch.autograd.grad((m(x) * t).sum(), [m.rho, m.phi, m.b], create_graph=True)
        got.append(torch.autograd.grad(sum((v * v).sum() for v in g), [m.rho, m.phi]))
    for a, b in zip(*got):
        assert torch.max(torch.abs(a - b)) <= 1e-12 * torch.max(torch.abs(b))


def test_host_parameters_keep_the_general_path():
    x, t = _signals()
    a, _ = _models()
    y = a(x)
    b, _ = _models()
    b = b.cpu()
    assert torch.equal(b(x), y)
