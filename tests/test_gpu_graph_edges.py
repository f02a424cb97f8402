"""Plans in a user's CUDA graph whose kernels are launched programmatically (a
cascade in phases; an FFT FIR of more than one wave of blocks): captured behind
a kernel that writes their input and before one that reads their output,
replayed on new inputs, to the bit what the same calls give one by one.  And
chains whose response needs the largest transform."""
import numpy as np
import pytest

from paper_2504_08624_gb300 import workloads as W
from tests.gpu_util import assert_close, oracle_chain

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _phases(S):
    rows = [[0.5, 0.0, 0.1, 1.0, -2 * 0.9995 * np.cos(0.3 + 0.4 * k), 0.9995 ** 2] for k in range(S)]
    return [("sos", np.array(rows))]


CASES = [("phase", 16, 131072, _phases(1)), ("phase", 16, 131072, _phases(2)), ("phase", 70, 131072, _phases(3)),
         ("fft", 64, 200000, [("fir", W.fir_lowpass(257, 9000.0, W.FS))]),
         ("fft", 33, 400001, [("sos", W.butter_sos(4, 1000.0, W.FS)), ("fir", W.fir_lowpass(1025, 9000.0, W.FS))]),
         ("fft", 32, 500000, [("fir", W.fir_bandpass(16384, 300.0, 3400.0, W.FS, ("kaiser", 8.0)))])]


@pytest.mark.parametrize("kind,C,Ns,stages", CASES)
def test_replayed_between_other_kernels(kind, C, Ns, stages):
    from paper_2504_08624_gb300 import api
    p = api.Plan(C, Ns, stages)
    d = p.describe()[0]
    if kind == "phase":
        assert d["scan"] == "phase"
    else:
        ctas = {4096: 8, 8192: 4, 16384: 2, 32768: 1}[d["M"]]
        assert d.get("P", 0) == 0 and C * (-(-Ns // d["B"])) > 152 * ctas, d
    src = [torch.from_numpy(W.white_gauss(C, Ns, 710 + i)).cuda() for i in range(3)]
    x, y, z = torch.empty_like(src[0]), torch.empty_like(src[0]), torch.empty_like(src[0])
    held = src[0].clone()

    def step():
        torch.mul(held, 2.0, out=x)
        p.execute(x, y)
        p.execute(y, x)  # the second call reads what the first writes
        torch.mul(x, -1.0, out=z)

    want = []
    for s in src:
        held.copy_(s)
        step()
        torch.cuda.synchronize()
        want.append(z.clone())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        step()
    for _ in range(2):
        for s, w in zip(src, want):
            held.copy_(s)
            z.zero_()
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(z, w)
    assert p.get_error() == 0
    p.close()


@pytest.mark.parametrize("fc,taps", [(17.0, 513), (20.0, 4097)])
def test_chain_composed_at_the_largest_transform(fc, taps):
    from paper_2504_08624_gb300 import api
    stages = [("sos", W.butter_sos(2, fc, W.FS)), ("fir", W.fir_lowpass(taps, 9000.0, W.FS))]
    x = W.white_gauss(16, 400003, 720)
    xd = torch.from_numpy(x).cuda()
    p = api.Plan(*x.shape, stages)
    d = p.describe()[0]
    assert d["kind"] == "chain_fft" and d["M"] == 32768 and d["Lc"] > 12289, d
    y = p.execute(xd, torch.empty_like(xd))
    torch.cuda.synchronize()
    assert p.get_error() == 0
    p.close()
    assert_close(y.cpu().numpy(), oracle_chain(x, stages), 1e-4, f"{d}")
