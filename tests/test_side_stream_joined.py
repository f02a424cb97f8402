"""A backward that fails after it has forked its side stream still joins it:
whatever already runs there is ordered before the caller's next work.  The
library runs on the CUDA runtime of fake_cudart.c (the host alone, no GPU),
whose n-th launch fails, for every n."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
import ctypes, importlib.util, json, sys
import numpy as np
root = sys.argv[1]
spec = importlib.util.spec_from_file_location("native", root + "/paper_2504_08624_gb300/_native.py")
N = importlib.util.module_from_spec(spec)
spec.loader.exec_module(N)
L, fake = N.lib(), ctypes.CDLL(None)
fake.fake_log.restype = ctypes.c_char_p
rows = np.array([[0.2, 0.1, 0.0, 1.0, -0.9, 0.3], [0.3, 0.0, 0.1, 1.0, -0.5, 0.2]])
st = N.StageList([("sos", rows), ("fir", np.full(33, 0.03))])
plan = ctypes.c_void_p()
C, Ns = 3, 6000
assert L.tfx_plan_create(ctypes.byref(plan), C, Ns, Ns, st.arr, st.n, N.TFX_PLAN_TRAINABLE) == 0
need = max(L.tfx_plan_backward_workspace_size(plan), L.tfx_plan_workspace_size(plan), 256)
buf = [np.zeros(C * Ns + 64, np.float32) for _ in range(5)]
x, y, t, g, dx = (ctypes.c_void_p(b.ctypes.data) for b in buf)
dc, loss = np.zeros(64), np.zeros(1)
room = np.zeros(need + 256, np.uint8)
ws = ctypes.c_void_p(room.ctypes.data + -room.ctypes.data % 256)
f64 = ctypes.POINTER(ctypes.c_double)
dcp, lp, stream = dc.ctypes.data_as(f64), loss.ctypes.data_as(f64), ctypes.c_void_p(64)
def step():
    return L.tfx_plan_train_step_mse(plan, x, y, t, g, lp, dx, dcp, ws, 0, ws, need, stream)
def backward():
    return L.tfx_plan_backward(plan, x, g, dx, ctypes.cast(dcp, ctypes.c_void_p), ws, 0, ws, need, stream)
out = []
for name, call in (("step", step), ("backward", backward)):
    for fail in range(0, 12):
        fake.fake_reset(fail)
        rc = call()
        out.append([name, fail, rc, fake.fake_log().decode()])
print(json.dumps(out))
"""


@pytest.fixture(scope="module")
def runs(tmp_path_factory):
    if not os.path.exists(os.path.join(ROOT, "paper_2504_08624_gb300", "_lib", "libtfx.so")):
        pytest.skip("libtfx.so has not been built")
    so = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", so, os.path.join(ROOT, "tests", "fake_cudart.c")], check=True)
    r = subprocess.run([sys.executable, "-c", PROGRAM, ROOT], env={**os.environ, "LD_PRELOAD": so}, capture_output=True,
                       text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    return json.loads(r.stdout)


def _unjoined(log, caller=64):
    """Streams with a launch that nothing orders before the caller's stream."""
    open_, events = set(), {}
    for line in log.splitlines():
        what, a, b = line.split()
        a, b = int(a), int(b)
        if what in ("launch", "copy") and a != caller:
            open_.add(a)
        elif what == "record":
            events[a] = b
        elif what == "wait" and a == caller and b in events:
            open_.discard(events[b])
    return open_


def test_every_failed_launch_leaves_the_side_stream_joined(runs):
    beside = False
    total = {name: sum(line.startswith("launch") for line in log.splitlines()) for name, fail, _, log in runs if not fail}
    for name, fail, rc, log in runs:
        assert (rc == 0) == (fail == 0 or fail > total[name]), (name, fail, rc, log)
        assert not _unjoined(log), (name, fail, rc, log)
        beside = beside or any(line.startswith("launch") and line.split()[1] != "64" for line in log.splitlines())
    assert beside and any(rc != 0 for _, _, rc, _ in runs)
