"""Executions of one batch on two streams stay independent: while the first
stream still waits for earlier work of its own, an execution on the second
one completes.  Outputs of both are those of an execution alone."""
import pytest

from .test_gpu_batch_beside import _batch, _same

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_a_blocked_caller_blocks_nobody():
    b, x, y = _batch()
    s = [torch.cuda.Stream() for _ in range(2)]
    ws = [torch.empty(b.workspace_size, dtype=torch.uint8, device="cuda") for _ in s]
    out = [torch.zeros_like(x) for _ in s]
    torch.cuda.synchronize()
    for first in range(2):  # whichever of them had the batch's stream before
        a = s[first]
        with torch.cuda.stream(a):
            torch.cuda._sleep(600_000_000)  # about 0.3 s
            b.execute(x, out[first], ws[first])
            done = torch.cuda.Event()
            done.record()
        other = 1 - first
        with torch.cuda.stream(s[other]):
            b.execute(x, out[other], ws[other])
        s[other].synchronize()
        alone = not done.query()
        assert _same(b, out[other], y)
        torch.cuda.synchronize()
        assert _same(b, out[first], y)
        assert alone
    assert b.get_error() == 0
    b.close()


def test_another_threads_capture_goes_on():
    """An execution that asks whether the batch's stream is free leaves a capture
    that another thread has under way (in the default, strictest mode) intact."""
    import threading
    b, x, y = _batch()
    s = [torch.cuda.Stream() for _ in range(2)]
    ws = [torch.empty(b.workspace_size, dtype=torch.uint8, device="cuda") for _ in s]
    out = [torch.zeros_like(x) for _ in s]
    v = torch.ones(1000, device="cuda")
    torch.cuda.synchronize()
    failed = []

    def run():
        try:
            with torch.cuda.stream(s[1]):
                b.execute(x, out[1], ws[1])
        except Exception as e:  # noqa: BLE001
            failed.append(e)

    with torch.cuda.stream(s[0]):
        b.execute(x, out[0], ws[0])
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        v.add_(1.0)
        t = threading.Thread(target=run)
        t.start()
        t.join()
        v.add_(1.0)
    torch.cuda.synchronize()
    assert not failed and _same(b, out[0], y) and _same(b, out[1], y)
    v.zero_()
    g.replay()
    assert bool((v == 2.0).all())
    b.close()
