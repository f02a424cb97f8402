"""A batch's composed clips at the largest transform, by choice of the caller
(fft_m of a length bucket) and as clip_info reports it."""
import numpy as np
import pytest

from paper_2504_08624_gb300 import workloads as W
from tests.gpu_util import assert_close, oracle_chain

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_fft_m_15():
    from paper_2504_08624_gb300 import api
    st = [("sos", W.butter_sos(4, 1000.0, W.FS)), ("fir", W.fir_lowpass(4097, 9000.0, W.FS))]
    clips = [(2, 70001, st), (1, 30000, st)]
    b = api.Batch(clips, fft_m={12: 15})
    xs = [W.white_gauss(C, Ns, 640 + i) for i, (C, Ns, _) in enumerate(clips)]
    x = b.empty()
    for i, v in enumerate(xs):
        assert b.clip_info(i)[0] and b.clip_info(i)[2] == 15
        b.view(x, i).copy_(torch.from_numpy(v))
    y = b.execute(x, torch.full_like(x, -7.0))
    torch.cuda.synchronize()
    assert b.get_error() == 0
    for i, v in enumerate(xs):
        assert_close(b.view(y, i).cpu().numpy().astype(np.float64), oracle_chain(v, st), 1e-4, str(clips[i][:2]))
    b.close()
