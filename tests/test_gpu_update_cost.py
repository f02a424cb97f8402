"""Coefficient updates of FFT FIRs and of spectral training plans: the tables
that the device forms filter as those of a new plan, and forming them takes
about as long as the transform that it needs (device time of a replayed graph
of updates; the bounds are about twice what an update by two blocks per
complex transform takes, and half or less of what FP64 trigonometry in one CTA
takes)."""
import numpy as np
import pytest

from paper_2504_08624_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _us(f, n=20):
    """Device time of one f() in a graph of n, the least of five replays."""
    f()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for _ in range(n):
            f()
    best = 1e9
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        g.replay()
        a.record()
        g.replay()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / n * 1e3)
    return best


@pytest.mark.parametrize("taps,C,N,bound", [(129, 8, 480000, 12.0), (1025, 8, 480000, 14.0), (2500, 8, 480000, 30.0),
                                            (4097, 8, 480000, 32.0), (12000, 8, 960000, 45.0), (16384, 8, 960000, 55.0)])
def test_fir_update(taps, C, N, bound):
    from paper_2504_08624_gb300 import api
    rng = np.random.default_rng(taps)
    h0, h1 = (rng.normal(0.0, taps ** -0.5, taps) for _ in range(2))
    p, q = api.Plan(C, N, [("fir", h0)]), api.Plan(C, N, [("fir", h1)])
    c = torch.from_numpy(h1).cuda()
    p.update_coefs(c)
    g = torch.Generator(device="cuda")
    g.manual_seed(taps)
    x = torch.randn(C, N, device="cuda", generator=g)
    a, b = p.execute(x, torch.empty_like(x)), q.execute(x, torch.empty_like(x))
    # both tables are within a few units of 2^-24 of the exact one
    assert torch.max(torch.abs(a - b)) <= 4e-6 * torch.max(torch.abs(b))
    took = _us(lambda: p.update_coefs(c))
    assert took <= bound, took


def test_input_gradient_after_an_update():
    """dL/dx of a spectral plan: after an update to the coefficients of another
    plan it is that plan's, for both transform sizes and odd section counts."""
    from paper_2504_08624_gb300 import _native as N_
    from paper_2504_08624_gb300 import api
    for S, taps, Ns in ((3, 129, 30001), (6, 2500, 40000)):
        def stages(seed):
            d = W.differentiable_chain_params(seed, S, taps)
            return [("sos", W.biquad_rows(d["rho"], d["phi"], d["b"])), ("fir", d["h"])]
        p, q = (api.Plan(4, Ns, stages(s), flags=N_.TFX_PLAN_TRAINABLE) for s in (41, 42))
        assert p.describe()[0]["kind"] == "chain_spectral"
        c = torch.cat([torch.from_numpy(np.ascontiguousarray(v)).reshape(-1) for _, v in stages(42)]).cuda()
        p.update_coefs(c)
        gen = torch.Generator(device="cuda")
        gen.manual_seed(S)
        x, g = (torch.randn(4, Ns, device="cuda", generator=gen) for _ in range(2))
        dx = []
        for k in (p, q):
            saved, y, d = k.new_saved(), torch.empty_like(x), torch.empty_like(x)
            k.forward_train(x, y, saved)
            k.backward(x, g, d, None, saved)
            dx.append(d)
        assert torch.max(torch.abs(dx[0] - dx[1])) <= 4e-6 * torch.max(torch.abs(dx[1]))
