"""Real blocks over rows at odd addresses: such a row's blocks start one
sample early, so that its samples move as pairs too.  Lengths at which that
takes one more block, an even row's last block is then empty, or a row has no
whole window at all; input and output odd together and apart; every transform
size; and the same in a batch, whose clips lie at odd offsets.  Tolerances:
1e-5 of each channel's peak, as for every FIR-only chain, and 1e-4, as for
every chain with sections."""
import numpy as np
import pytest

from paper_2504_08624_gb300 import workloads as W
from tests.gpu_util import assert_close, oracle_chain
from tests.test_gpu_real_blocks import _check, _taps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [12, 13, 14])
@pytest.mark.parametrize("xoff,yoff,pad", [(1, 1, 0), (0, 0, 1), (1, 0, 1), (0, 1, 1), (3, 1, 2)])
def test_lengths_around_the_blocks(m, xoff, yoff, pad):
    M = 1 << m
    L = M // 4 + 1
    B = M - M // 4
    for Ns in (1, B - 1, B, 2 * B - 1, 2 * B, 3 * B + 7):
        d = _check(W.white_gauss(3, Ns, 950 + Ns % 83), _taps(L, m), m=m, xoff=xoff, yoff=yoff, pad=pad)
        assert d["M"] == M and d["B"] == B and d["P"] == 0


@pytest.mark.parametrize("Ns", [65536, 65535])
@pytest.mark.parametrize("xoff,yoff,pad", [(1, 1, 0), (0, 0, 1), (0, 1, 1)])
def test_largest_block(Ns, xoff, yoff, pad):
    d = _check(W.white_gauss(4, Ns, 960), _taps(16384, 3), xoff=xoff, yoff=yoff, pad=pad)
    assert d["M"] == 32768 and d["B"] == 16384


def test_batch_clips_at_odd_offsets():
    from paper_2504_08624_gb300 import api
    st = [("sos", W.butter_sos(4, 1000.0, W.FS)), ("fir", W.fir_lowpass(257, 9000.0, W.FS))]
    b = api.Batch([(1, 40001, st)])
    composed, L, m = b.clip_info(0)
    b.close()
    assert composed and m >= 12
    B = (1 << m) - (L - 1 + (L - 1) % 2)
    # an odd clip first, so that the rows after it start odd; then both kinds of row
    clips = [(1, 8 * B + 1, st), (2, 4 * B, st), (3, 5 * B - 1, st), (1, 8 * B, st), (2, 6 * B + 1, st)]
    b = api.Batch(clips)
    xs = [W.white_gauss(C, Ns, 970 + i) for i, (C, Ns, _) in enumerate(clips)]
    x = b.empty()
    for i, v in enumerate(xs):
        assert b.clip_info(i) == (True, L, m)
        b.view(x, i).copy_(torch.from_numpy(v))
    y = b.execute(x, torch.full_like(x, -7.0))
    torch.cuda.synchronize()
    assert b.get_error() == 0
    for i, v in enumerate(xs):
        assert_close(b.view(y, i).cpu().numpy().astype(np.float64), oracle_chain(v, st), 1e-4, str(clips[i][:2]))
    b.close()
