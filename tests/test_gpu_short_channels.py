"""Many short channels, and signals of few blocks: a block never spans two
channels, so the transform size follows the channel's length, and a signal that
one wave of blocks holds takes the size of least latency (real blocks of 1024 and
2048 samples, which longer signals do not take, included).  Which size a plan takes, and those two
sizes against the oracle at lengths around a block, at odd addresses, after a
coefficient update, in place and in a batch.  Tolerances: 1e-5 of each channel's
peak, as for every FIR-only chain, and 1e-4, as for every chain with sections."""
import numpy as np
import pytest

from paper_2504_08624_gb300 import workloads as W
from tests.gpu_util import assert_close, oracle_chain
from tests.test_gpu_real_blocks import _check, _taps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,taps,N,M", [
    (4096, 65, 300, 1024), (4096, 129, 1900, 2048), (4096, 257, 600, 1024), (4096, 513, 3000, 4096),
    (4096, 1025, 3000, 4096), (4096, 2049, 6000, 8192), (4096, 65, 16383, 2048), (4096, 65, 16384, 4096),
    (1, 65, 24000, 2048), (1, 2011, 24001, 4096), (16, 65, 25000, 2048), (8, 4097, 50000, 8192),
    (64, 2011, 1000000, 16384), (5, 5231, 250000, 16384), (4, 12290, 81907, 32768)])
def test_size_follows_the_signal(C, taps, N, M):
    from paper_2504_08624_gb300 import api
    p = api.Plan(C, N, [("fir", _taps(taps, 1))])
    d = p.describe()[0]
    p.close()
    assert d["kind"] == "fir_fft" and d["P"] == 0 and d["M"] == M, d


def test_composed_chain_and_long_signals():
    from paper_2504_08624_gb300 import api
    st = [("sos", W.butter_sos(4, 1000.0, W.FS))]
    long = api.Plan(64, 1000000, st).describe()[0]
    assert long["kind"] == "chain_fft" and long["M"] == 4096
    J = long["Lc"] - 1 + (long["Lc"] - 1) % 2
    assert 256 < J < 512
    for C, N, M in ((8, 1000, 2048), (8, 6000, 2048), (4096, 2048 - J, 2048), (4096, 4096 - J, 4096)):
        d = api.Plan(C, N, st).describe()[0]
        assert d["kind"] == "chain_fft" and d["Lc"] == long["Lc"] and d["M"] == M, d


@pytest.mark.parametrize("m", [10, 11])
@pytest.mark.parametrize("even", [False, True])
def test_lengths_around_a_block(m, even):
    M = 1 << m
    L = M // 4 + (2 if even else 1)
    B = M - (L - 1 + (L - 1) % 2)
    for xoff, yoff, pad in ((0, 0, 0), (1, 1, 0), (0, 0, 1), (1, 0, 1), (0, 1, 0), (2, 3, 2)):
        for Ns in (1, 2, B - 1, B, B + 1, 2 * B - 1, 3 * B + 2):
            d = _check(W.white_gauss(3, Ns, 600 + Ns % 89), _taps(L, m), m=m, xoff=xoff, yoff=yoff, pad=pad)
            assert d["M"] == M and d["B"] == B and d["P"] == 0


@pytest.mark.parametrize("L,N", [(65, 301), (257, 1001), (513, 2999), (64, 700)])
def test_many_channels_in_place_and_updated(L, N):
    from paper_2504_08624_gb300 import api
    h = _taps(L, L)
    x = W.white_gauss(700, N, 610)
    want = oracle_chain(x, [("fir", h)])
    for update in (False, True):
        p = api.Plan(700, N, [("fir", _taps(L, 3) if update else h)])
        assert p.describe()[0]["M"] <= (2048 if L < 513 else 4096)
        if update:
            p.update_coefs(torch.from_numpy(h).cuda())
        xd = torch.from_numpy(x).cuda()
        y = p.execute(xd, torch.empty_like(xd))
        p.execute(xd, xd)
        assert torch.equal(xd, y)
        assert_close(y.cpu().numpy().astype(np.float64), want, 1e-5, f"{L} {N} {update}")
        p.close()


def _batch(clips, **kw):
    """Runs the clips in a batch, each checked against the oracle; their sizes."""
    from paper_2504_08624_gb300 import api
    b = api.Batch(clips, **kw)
    xs = [W.white_gauss(C, Ns, 620 + i % 97) for i, (C, Ns, _) in enumerate(clips)]
    x = b.empty()
    for i, v in enumerate(xs):
        b.view(x, i).copy_(torch.from_numpy(v))
    y = b.execute(x, torch.full_like(x, -7.0))
    torch.cuda.synchronize()
    assert b.get_error() == 0
    for i, v in enumerate(xs):
        assert_close(b.view(y, i).cpu().numpy().astype(np.float64), oracle_chain(v, clips[i][2]), 1e-4, str(clips[i][:2]))
    info = [b.clip_info(i) for i in range(len(clips))]
    groups = [(k, lev) for k, lev, *_ in b.groups()]
    b.close()
    return info, groups


SOS = ("sos", W.butter_sos(4, 1000.0, W.FS))
R, TH = 0.9995, 0.3  # its units stay
SLOW = ("sos", np.array([[1e-4, 0.0, -1e-4, 1.0, -2 * R * np.cos(TH), R * R]]))


def _fir(L):
    return ("fir", W.fir_lowpass(L, 9000.0, W.FS))


def test_batch_of_short_clips():
    """One common size, one launch: composed clips, and FIRs of two levels."""
    info, groups = _batch([(1 + i % 3, 1001 + 7 * i, [SOS] + ([_fir(65)] if i % 2 else [])) for i in range(120)])
    assert all(c and m == info[0][2] <= 11 for c, _, m in info) and [k for k, _ in groups] == [3]
    clips = [(2, 701 + 3 * i, [_fir(65 + 64 * (i % 2)), SLOW]) for i in range(80)]
    clips += [(1, 1500 + i, [SLOW, _fir(257)]) for i in range(80)]
    info, groups = _batch(clips)
    assert not any(c for c, _, _ in info) and sum(k == 4 for k, _ in groups) == 2


def test_batch_of_short_and_long_clips():
    """Long clips keep their size; a few short ones stay with them, many get a
    launch of their own; a size that the caller gave stays."""
    long = [(2, 200001, [SOS])]
    few = [(3, 1001, [SOS]), (1, 2500, [SOS, _fir(129)])]
    info, groups = _batch(long + few)
    assert [m for _, _, m in info] == [12, 12, 12] and len(groups) == 1
    many = [(40, 801 + i, [SOS]) for i in range(40)]
    info, groups = _batch(long + many)
    assert info[0][2] == 12 and all(m < 12 for _, _, m in info[1:]) and len(groups) == 2
    info, _ = _batch(long + many[:10], fft_m={8: 13})
    assert all(m == 13 for _, _, m in info)
