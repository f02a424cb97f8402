"""An infinity or a NaN in one sample: rows that do not hold it are untouched
(to the bit), and in its own row everything outside the outputs that the route
computes from it: a cascade in phases changes nothing before it, a direct FIR
nothing from L + 3 samples after it on (taps are padded to a multiple of four),
an FFT FIR nothing a whole transform away."""
import numpy as np
import pytest

from paper_2504_08624_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BAD = [float("nan"), float("inf"), float("-inf")]


def _outputs(stages, C, Ns, row, at, bad, pad=0, flags=0):
    """(clean, touched) outputs of one plan, and its description."""
    from paper_2504_08624_gb300 import api
    p = api.Plan(C, Ns, stages, ld=Ns + pad, flags=flags)
    x = torch.empty((C, Ns + pad), device="cuda")[:, :Ns]
    x.copy_(torch.from_numpy(W.white_gauss(C, Ns, 701)))
    out = []
    for v in (None, bad):
        if v is not None:
            x[row, at] = v
        y = torch.empty((C, Ns + pad), device="cuda")[:, :Ns]
        out.append(p.execute(x, y).clone())
    torch.cuda.synchronize()
    assert p.get_error() == 0
    d = p.describe()[0]
    p.close()
    clean, touched = out
    assert torch.isfinite(clean).all() and not torch.isfinite(touched[row, at])
    rest = [c for c in range(C) if c != row]
    assert torch.equal(clean[rest], touched[rest])
    return clean[row], touched[row], d


@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("at", [0, 1000, 8191, 8192, 70001])
def test_cascade_in_phases(bad, at):
    rows = np.array([[0.5, 0.0, 0.1, 1.0, -2 * 0.9995 * np.cos(0.3), 0.9995 ** 2]])
    a, b, d = _outputs([("sos", np.concatenate([rows, W.butter_sos(2, 3000.0, W.FS)]))], 16, 131073, 5, at, bad)
    assert d["scan"] == "phase" and torch.equal(a[:at], b[:at])


@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("L", [1, 33, 63])
@pytest.mark.parametrize("at", [0, 2047, 2048, 9000])
def test_direct_fir(bad, L, at):
    a, b, d = _outputs([("fir", np.linspace(1.0, 0.5, L))], 3, 9011, 1, at, bad, pad=2)
    assert d["kind"] == "fir" and torch.equal(a[:at], b[:at]) and torch.equal(a[at + L + 3:], b[at + L + 3:])


@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("m", [10, 11, 12, 13, 14])
def test_fft_fir(bad, m):
    from paper_2504_08624_gb300 import _native as N_
    M = 1 << m
    for pad in (0, 1):
        a, b, d = _outputs([("fir", W.fir_lowpass(101, 9000.0, W.FS))], 3, 5 * M + 3, 1, 2 * M + 7, bad, pad=pad,
                           flags=N_.TFX_PLAN_FIR_FFT | N_.TFX_PLAN_FIR_FFT_LOG(m))
        assert d["M"] == M and d["P"] == 0
        assert torch.equal(a[:M + 7], b[:M + 7]) and torch.equal(a[3 * M + 7:], b[3 * M + 7:])
