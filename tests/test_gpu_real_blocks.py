"""Single-block overlap-save with one real block per transform (k_fir_rfft):
M = 4096, 8192, 16384 and 32768 samples.  Windows move as pairs of samples
where a row starts on an 8-byte boundary and as single samples elsewhere, and
blocks at a channel's ends read and write part of a window: both are run here
against the oracle, at lengths around a block, with even and odd tap counts
(the overlap is rounded up to even), odd strides and odd base addresses of
the input and of the output separately.  Tolerance: 1e-5 of each channel's
peak, as for every FIR-only chain."""
import math

import numpy as np
import pytest

from paper_2504_08624_gb300 import workloads as W
from tests.gpu_util import assert_close, oracle_chain

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _taps(L, seed):
    return np.random.default_rng(seed).standard_normal(L) / math.sqrt(L)


def _run(x, h, m=None, xoff=0, yoff=0, pad=0, update=False):
    """The filter through a plan of transform size 2^m (None: the model's),
    input and output starting xoff and yoff floats after an aligned address."""
    from paper_2504_08624_gb300 import _native as N_
    from paper_2504_08624_gb300 import api
    C, Ns = x.shape
    ld = Ns + pad
    flags = N_.TFX_PLAN_FIR_FFT | (N_.TFX_PLAN_FIR_FFT_LOG(m) if m else 0)
    first = _taps(len(h), 99) if update else h
    p = api.Plan(C, Ns, [("fir", first)], ld=ld, flags=flags)
    d = p.describe()[0]
    if update:
        p.update_coefs(torch.from_numpy(np.asarray(h, dtype=np.float64)).cuda())
    xb = torch.full((C * ld + 8,), 3.0, device="cuda")
    yb = torch.full((C * ld + 8,), -7.0, device="cuda")
    xv, yv = (b[o:o + C * ld].view(C, ld)[:, :Ns] for b, o in ((xb, xoff), (yb, yoff)))
    xv.copy_(torch.from_numpy(x))
    p.execute(xv, yv)
    torch.cuda.synchronize()
    assert p.get_error() == 0
    p.close()
    keep = torch.ones_like(yb, dtype=torch.bool)
    keep[yoff:yoff + C * ld].view(C, ld)[:, :Ns] = False
    assert torch.all(yb[keep] == -7.0)  # nothing but the rows is written
    return yv.cpu().numpy().astype(np.float64), d


def _check(x, h, **kw):
    got, d = _run(x, h, **kw)
    assert_close(got, oracle_chain(x, [("fir", h)]), 1e-5, f"{d} {kw}")
    return d


@pytest.mark.parametrize("m", [12, 13, 14])
@pytest.mark.parametrize("even", [False, True])
def test_lengths_around_a_block(m, even):
    M = 1 << m
    L = M // 4 + (2 if even else 1)
    B = M - (L - 1 + (L - 1) % 2)
    for Ns in (1, 2, B - 1, B, B + 1, 3 * B + 2):
        d = _check(W.white_gauss(2, Ns, 900 + Ns % 89), _taps(L, m), m=m)
        assert d["M"] == M and d["B"] == B and d["P"] == 0


@pytest.mark.parametrize("m", [12, 13, 14])
@pytest.mark.parametrize("xoff,yoff,pad", [(0, 0, 1), (1, 0, 0), (0, 1, 0), (1, 1, 3), (2, 3, 2)])
def test_unaligned_rows(m, xoff, yoff, pad):
    x = W.white_gauss(3, 40001, 910)
    _check(x, _taps(300, 5), m=m, xoff=xoff, yoff=yoff, pad=pad)


def test_largest_block():
    """M = 32768: taps beyond the 16384-sample blocks, from 16 blocks on; one
    block fewer keeps the partitioned scheme."""
    for L in (12290, 16384, 20000):
        B = 32768 - (L - 1 + (L - 1) % 2)
        d = _check(W.white_gauss(4, 4 * B - 5, 920), _taps(L, L), pad=1)
        assert d["M"] == 32768 and d["B"] == B and d["P"] == 0
    d = _check(W.white_gauss(3, 5 * 16384, 921), _taps(16384, 1))
    assert d["P"] > 0


@pytest.mark.parametrize("m,L", [(12, 1000), (13, 2049), (14, 4097), (None, 16384)])
def test_taps_updated_on_the_device(m, L):
    x = W.white_gauss(8, 40000 if m else 3 * 16384, 930)
    d = _check(x, _taps(L, 7), m=m, update=True)
    assert d["P"] == 0


def test_short_and_single_taps():
    """Taps far below the block, down to the shortest the route takes."""
    x = W.white_uniform(3, 20011, 940)
    for L in (64, 65):
        _check(x, _taps(L, L))
    one = np.zeros(64)
    one[0] = 1.0  # the unit impulse returns the signal
    got, _ = _run(x, one)
    assert np.max(np.abs(got - x)) <= 1e-5
