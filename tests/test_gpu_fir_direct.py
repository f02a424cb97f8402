"""Short FIRs alone (k_fir_direct: 1 to 63 taps, independent tiles of 2048
outputs that start on 16-byte boundaries of the row) against the oracle:
lengths around a tile, tap counts around the kernel's steps of 4 and 16, odd
strides, odd base addresses of the input and of the output, one sample, and
the in-place call (which keeps the tile-to-tile kernel).  Tolerance: 1e-5 of
each channel's peak."""
import numpy as np
import pytest

from paper_2504_08624_gb300 import workloads as W
from tests.gpu_util import assert_close, oracle_chain

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(C, Ns, L, xoff=0, yoff=0, pad=0, inplace=False):
    from paper_2504_08624_gb300 import api
    x = W.white_gauss(C, Ns, 1000 + Ns % 83)
    h = np.random.default_rng(L).standard_normal(L) / np.sqrt(L)
    ld = Ns + pad
    xb = torch.full((C * ld + 8,), 3.0, device="cuda")
    yb = xb if inplace else torch.full((C * ld + 8,), -7.0, device="cuda")
    if inplace:
        yoff = xoff
    xv, yv = (b[o:o + C * ld].view(C, ld)[:, :Ns] for b, o in ((xb, xoff), (yb, yoff)))
    xv.copy_(torch.from_numpy(x))
    p = api.Plan(C, Ns, [("fir", h)], ld=ld)
    p.execute(xv, yv)
    torch.cuda.synchronize()
    assert p.get_error() == 0
    p.close()
    keep = torch.ones_like(yb, dtype=torch.bool)
    keep[yoff:yoff + C * ld].view(C, ld)[:, :Ns] = False
    assert torch.all(yb[keep] == (3.0 if inplace else -7.0))
    assert_close(yv.cpu().numpy().astype(np.float64), oracle_chain(x, [("fir", h)]), 1e-5, f"{C}x{Ns}, {L} taps")


@pytest.mark.parametrize("L", [1, 3, 4, 5, 16, 17, 32, 33, 48, 49, 63])
def test_tap_counts(L):
    for Ns in (1, 5, 2045, 2048, 2049, 6147):
        _check(2, Ns, L)


@pytest.mark.parametrize("xoff,yoff,pad", [(0, 0, 1), (1, 0, 0), (0, 1, 0), (3, 3, 2), (2, 1, 3)])
def test_unaligned_rows(xoff, yoff, pad):
    for Ns in (2, 2047, 20001):
        _check(3, Ns, 33, xoff=xoff, yoff=yoff, pad=pad)


def test_in_place():
    _check(3, 20001, 33, xoff=1, pad=2, inplace=True)
