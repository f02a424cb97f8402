"""A batch whose groups run beside one another (composed clips of several
transform sizes and clips that keep their units): its outputs in
executions from two threads on two streams, from a replayed graph, and while
another thread captures the same batch."""
import threading

import numpy as np
import pytest

from paper_2504_08624_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _batch():
    from paper_2504_08624_gb300 import api
    r, th = 0.9995, 0.3  # does not compose: its cascade and FIR stay units
    slow = [("sos", np.array([[1e-4, 0.0, -1e-4, 1.0, -2 * r * np.cos(th), r * r]])), ("fir", W.fir_lowpass(65, 9000.0, W.FS))]
    clips = [(2, 60000, slow), (3, 50001, slow)]
    clips += [(2, 90000, [("sos", W.butter_sos(4, 1000.0, W.FS)), ("fir", W.fir_lowpass(L, 9000.0, W.FS))])
              for L in (33, 1025, 4097)]
    b = api.Batch(clips)
    assert len(b.groups()) >= 4 and not b.clip_info(0)[0] and b.clip_info(2)[0]
    x = b.empty().uniform_(-1.0, 1.0)
    y = b.execute(x, torch.zeros_like(x), torch.empty(b.workspace_size, dtype=torch.uint8, device="cuda"))
    torch.cuda.synchronize()
    return b, x, y


def _same(b, got, want):
    """Composed clips to the bit; the units' look-back adds its carries in the
    order the tiles finish, so those clips to the cascades' tolerance."""
    for i in range(len(b.clips)):
        g, w = b.view(got, i), b.view(want, i)
        if b.clip_info(i)[0]:
            if not torch.equal(g, w):
                return False
        elif not bool((g - w).abs().max() <= 1e-4 * w.abs().max()):
            return False
    return True


def test_two_threads():
    b, x, y = _batch()
    bad = []

    def run():
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            ws = torch.empty(b.workspace_size, dtype=torch.uint8, device="cuda")
            for _ in range(20):
                out = torch.zeros_like(x)
                b.execute(x, out, ws)
                s.synchronize()
                if not _same(b, out, y):
                    bad.append(1)

    th = [threading.Thread(target=run) for _ in range(2)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not bad and b.get_error() == 0
    b.close()


def test_capture_beside_executions():
    b, x, y = _batch()
    ws = [torch.empty(b.workspace_size, dtype=torch.uint8, device="cuda") for _ in range(2)]
    out, eager = torch.zeros_like(x), torch.zeros_like(x)
    stop, bad = threading.Event(), []

    def run():
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            while not stop.is_set():
                b.execute(x, eager, ws[1])
                s.synchronize()
                if not _same(b, eager, y):
                    bad.append(1)

    t = threading.Thread(target=run)
    t.start()
    try:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, capture_error_mode="thread_local"):
            b.execute(x, out, ws[0])
            b.execute(x, out, ws[0])  # twice in one capture
    finally:
        stop.set()
        t.join()
    torch.cuda.synchronize()
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert _same(b, out, y) and not bad and b.get_error() == 0
    b.close()
