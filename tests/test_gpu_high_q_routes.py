"""Poles next to the unit circle through both forms of the FP64-carry cascade:
in phases (k_sos_phase, what long signals of up to four sections take) and by
look-back (k_sos_warp, what longer cascades, shorter signals, training plans and
the flag take).  Tolerance: 1e-4 of each channel's peak, as for every chain
with sections (FP64 carries measured 3.3e-5 at r = 0.99999)."""
import numpy as np
import pytest

from paper_2504_08624_gb300 import workloads as W
from tests.gpu_util import assert_close, oracle_chain
from tests.test_gpu_parity import _resonator

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rows(S, r, th):
    rows = [_resonator(r, th)]
    rows += [W.butter_sos(2, fc, 48000.0) for fc in (2000.0, 6000.0, 9000.0, 12000.0, 15000.0)]
    return np.concatenate(rows)[:S]


def _check(x, rows, scan, flags=0):
    from paper_2504_08624_gb300 import api
    xd = torch.from_numpy(x).cuda()
    p = api.Plan(*x.shape, [("sos", rows)], flags=flags)
    d = p.describe()
    assert [(u["S"], u["scan"], u["carry"]) for u in d] == [(len(rows), scan, "fp64")], d
    y = p.execute(xd, torch.empty_like(xd))
    torch.cuda.synchronize()
    assert p.get_error() == 0
    p.close()
    assert_close(y.cpu().numpy(), oracle_chain(x, [("sos", rows)]), 1e-4, f"{scan}, {len(rows)} sections")


@pytest.mark.parametrize("r", [0.9995, 0.9999, 0.99999])
@pytest.mark.parametrize("th", [0.05, 0.5])
@pytest.mark.parametrize("S", [1, 2])
def test_both_forms(r, th, S):
    from paper_2504_08624_gb300 import _native as N_
    x = W.white_uniform(2, 1 << 20, 77)
    _check(x, _rows(S, r, th), "phase")
    _check(x, _rows(S, r, th), "warp", N_.TFX_PLAN_SCAN_LOOKBACK)


@pytest.mark.parametrize("S", [3, 4])
@pytest.mark.parametrize("th", [0.05, 0.5])
def test_longer_cascades_in_phases(S, th):
    _check(W.white_uniform(1, 1 << 20, 79), _rows(S, 0.99999, th), "phase")


@pytest.mark.parametrize("th", [0.05, 0.5])
def test_more_sections_keep_the_look_back(th):
    _check(W.white_uniform(2, 1 << 20, 80), _rows(5, 0.99999, th), "warp")
