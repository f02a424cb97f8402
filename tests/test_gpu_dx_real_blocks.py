"""The input gradient of a spectral training plan, which runs as real blocks
over the rows in reverse time, against the oracle: lengths around a block,
even and odd, rows that start on odd addresses, both transform sizes, chains
with and without an FIR, one to many sections (the chain's product table takes
an even number of roots per warp), and after a coefficient update on the
device.  Tolerance: 1e-4 of each channel's peak, as for every chain with
sections."""
import numpy as np
import pytest

import oracle
from paper_2504_08624_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dx(stages, C, Ns, M, off=0, pad=0, update=None):
    from paper_2504_08624_gb300 import _native as N_
    from paper_2504_08624_gb300 import api
    ld = Ns + pad
    p = api.Plan(C, Ns, stages, ld=ld, flags=N_.TFX_PLAN_TRAINABLE)
    d = p.describe()[0]
    assert d["kind"] == "chain_spectral" and d["M"] == M, d
    if update is not None:
        p.update_coefs(torch.from_numpy(np.concatenate([np.asarray(c, dtype=np.float64).ravel() for _, c in update])).cuda())
    g = W.white_gauss(C, Ns, 1200 + Ns % 61)
    bufs = [torch.full((C * ld + 8,), v, device="cuda") for v in (0.0, 3.0, -7.0)]
    x, gv, dx = (b[off:off + C * ld].view(C, ld)[:, :Ns] for b in bufs)
    gv.copy_(torch.from_numpy(g))
    p.backward(x, gv, dx, None, p.new_saved())
    torch.cuda.synchronize()
    assert p.get_error() == 0
    p.close()
    keep = torch.ones_like(bufs[2], dtype=torch.bool)
    keep[off:off + C * ld].view(C, ld)[:, :Ns] = False
    assert torch.all(bufs[2][keep] == -7.0)
    # the transposed chain: the chain over the rows in reverse time
    ref = oracle.chain(np.ascontiguousarray(g[:, ::-1]), update or stages)[:, ::-1]
    got = dx.cpu().numpy().astype(np.float64)
    err = np.max(np.abs(got - ref), axis=1) / np.max(np.abs(ref), axis=1)
    assert np.all(err <= 1e-4), (d, err)


def _chain(S, taps, rmax=0.97):
    st = [("sos", W.random_stable_sos(S, 50 + S, 0.3, rmax))]
    return st + ([("fir", W.fir_lowpass(taps, 9000.0, W.FS))] if taps else [])


@pytest.mark.parametrize("S,taps", [(1, 0), (2, 33), (3, 0), (5, 257), (6, 257), (7, 64), (11, 0), (16, 9)])
def test_sections_and_taps(S, taps):
    _dx(_chain(S, taps, 0.9), 3, 9001, 4096)


@pytest.mark.parametrize("off,pad", [(0, 0), (1, 0), (0, 1), (1, 2)])
@pytest.mark.parametrize("Ns", [3072, 3073, 6144, 9215, 9216])
def test_lengths_and_rows(Ns, off, pad):
    _dx(_chain(4, 33, 0.9), 2, Ns, 4096, off, pad)


def test_larger_transform_and_update():
    stages = [("sos", W.random_stable_sos(3, 60, 0.3, 0.95)), ("fir", W.fir_lowpass(3001, 9000.0, W.FS))]
    _dx(stages, 3, 30001, 8192)
    new = [("sos", W.random_stable_sos(3, 61, 0.3, 0.95)), ("fir", W.fir_lowpass(3001, 5000.0, W.FS))]
    _dx(stages, 3, 30001, 8192, update=new)
    _dx(_chain(6, 257, 0.9), 4, 12000, 4096, update=_chain(6, 257, 0.85))
