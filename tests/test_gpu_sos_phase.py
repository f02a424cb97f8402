"""FP64-carry cascades in phases (k_sos_phase) against the oracle and the
look-back kernel: lengths around the 8192-sample tile and the 1024-sample warp
tile, one to four sections, odd strides and addresses, in place, and the sizes
from which the phases are taken.  Tolerance: 1e-4 of each channel's peak (the
poles' FP32 coefficients included, as for the look-back)."""
import numpy as np
import pytest

from paper_2504_08624_gb300 import workloads as W
from tests.gpu_util import assert_close, oracle_chain

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rows(S, r=0.9995):
    """Resonators of radius r at well separated angles, unit peak gain."""
    out = []
    for k in range(S):
        th = 0.3 + 0.5 * k
        w = np.exp(-1j * th)
        g = abs((1 - w * w) / (1 - 2 * r * np.cos(th) * w + r * r * w * w))
        out.append([1 / g, 0.0, -1 / g, 1.0, -2 * r * np.cos(th), r * r])
    # one after another they would cancel: mix with the signal (a notch's complement)
    return np.array([[b[0] + 0.5 * b[3], b[1] + 0.5 * b[4], b[2] + 0.5 * b[5], b[3], b[4], b[5]] for b in out])


def _run(C, Ns, S, xoff=0, yoff=0, pad=0, inplace=False, flags=0):
    from paper_2504_08624_gb300 import api
    stages = [("sos", _rows(S))]
    x = W.white_gauss(C, Ns, 1100 + Ns % 79)
    ld = Ns + pad
    xb = torch.full((C * ld + 8,), 3.0, device="cuda")
    yb = xb if inplace else torch.full((C * ld + 8,), -7.0, device="cuda")
    yoff = xoff if inplace else yoff
    xv, yv = (b[o:o + C * ld].view(C, ld)[:, :Ns] for b, o in ((xb, xoff), (yb, yoff)))
    xv.copy_(torch.from_numpy(x))
    p = api.Plan(C, Ns, stages, ld=ld, flags=flags)
    n = p.launches_per_execute
    p.execute(xv, yv)
    torch.cuda.synchronize()
    assert p.get_error() == 0
    p.close()
    keep = torch.ones_like(yb, dtype=torch.bool)
    keep[yoff:yoff + C * ld].view(C, ld)[:, :Ns] = False
    assert torch.all(yb[keep] == (3.0 if inplace else -7.0))
    assert_close(yv.cpu().numpy().astype(np.float64), oracle_chain(x, stages), 1e-4, f"{C}x{Ns}, {S} sections")
    return n


@pytest.mark.parametrize("Ns", [125000, 122880, 122881, 123903, 131071, 131073])
def test_lengths_around_a_tile(Ns):
    assert _run(9, Ns, 1) == 3


@pytest.mark.parametrize("S,C", [(2, 16), (3, 61), (4, 101)])
def test_sections(S, C):
    assert _run(C, 100003, S) == 2 * S + 1


@pytest.mark.parametrize("xoff,yoff,pad,inplace", [(0, 0, 1, False), (1, 2, 0, False), (3, 3, 2, True),
                                                   (0, 0, 0, True)])
def test_rows_and_in_place(xoff, yoff, pad, inplace):
    assert _run(9, 120000, 2 if pad else 1, xoff, yoff, pad, inplace) in (1, 3)
    assert _run(16, 120000, 2, xoff, yoff, pad, inplace) == 5


@pytest.mark.parametrize("tiles,C", [(32, 4), (64, 2), (128, 1)])
@pytest.mark.parametrize("more", [0, 1])
def test_tiles_around_the_threads_of_the_carry_scan(tiles, C, more):
    assert _run(C, 8192 * tiles + more, 1) == 3


@pytest.mark.parametrize("Ns", [24576, 24577, 32767, 40001])
def test_short_channels(Ns):
    assert _run(11, Ns, 1) == 3


def test_sizes_that_keep_the_look_back():
    assert _run(16, 24575, 1) == 1
    assert _run(5, 49999, 1) == 1
    assert _run(5, 50000, 1) == 3
    assert _run(1, 199999, 2) == 1
    assert _run(1, 200000, 2) == 5


@pytest.mark.parametrize("flag", ["TFX_PLAN_SCAN_LOOKBACK", "TFX_PLAN_SCAN_WARP_TILES"])
def test_asked_for_look_back(flag):
    from paper_2504_08624_gb300 import _native as N_
    assert _run(2, 500000, 1, flags=getattr(N_, flag)) == 1
