"""What the FFT tables of a size hold whatever the filter is formed once: a
further plan of that size takes no sines and cosines for it, from whichever
thread, and its constants are the first one's.  The library runs on the CUDA
runtime of fake_cudart.c (the host alone), with sin, cos and sincos counted."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

COUNT = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdatomic.h>
static atomic_long n;
long trig_calls(void) { return n; }
double sin(double x) { static double (*f)(double); if (!f) f = dlsym(RTLD_NEXT, "sin"); ++n; return f(x); }
double cos(double x) { static double (*f)(double); if (!f) f = dlsym(RTLD_NEXT, "cos"); ++n; return f(x); }
void sincos(double x, double *s, double *c) {
    static void (*f)(double, double *, double *);
    if (!f) f = dlsym(RTLD_NEXT, "sincos");
    ++n;
    f(x, s, c);
}
"""

PROGRAM = r"""
import ctypes, importlib.util, json, sys, threading
import numpy as np
root = sys.argv[1]
spec = importlib.util.spec_from_file_location("native", root + "/paper_2504_08624_gb300/_native.py")
N = importlib.util.module_from_spec(spec)
spec.loader.exec_module(N)
L, fake = N.lib(), ctypes.CDLL(None)
fake.trig_calls.restype = ctypes.c_long
fake.fake_last_upload.restype = ctypes.c_char_p
h = N.StageList([("fir", np.linspace(1.0, 0.5, 65))])
def plan(m):
    p = ctypes.c_void_p()
    before = fake.trig_calls()
    assert L.tfx_plan_create(ctypes.byref(p), 2, 100000, 100000, h.arr, h.n, N.TFX_PLAN_FIR_FFT | N.TFX_PLAN_FIR_FFT_LOG(m)) == 0
    return fake.trig_calls() - before, fake.fake_last_upload().decode()
out = {}
for m in (10, 11, 12, 13, 14):
    out[m] = [plan(m), plan(m)]
    got = []
    th = [threading.Thread(target=lambda: got.append(plan(m)[0])) for _ in range(4)]
    for t in th: t.start()
    for t in th: t.join()
    out[m] += [[sum(got), out[m][0][1]]]
print(json.dumps(out))
"""


def test_second_plan_takes_no_trigonometry(tmp_path):
    if not os.path.exists(os.path.join(ROOT, "paper_2504_08624_gb300", "_lib", "libtfx.so")):
        pytest.skip("libtfx.so has not been built")
    src, so = tmp_path / "count.c", str(tmp_path / "libfake.so")
    src.write_text(COUNT)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-fno-builtin", "-o", so, os.path.join(ROOT, "tests", "fake_cudart.c"),
                    str(src), "-ldl"], check=True)
    r = subprocess.run([sys.executable, "-c", PROGRAM, ROOT], env={**os.environ, "LD_PRELOAD": so}, capture_output=True,
                       text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    for m, runs in json.loads(r.stdout).items():
        (first, a), (second, b), (threads, _) = runs
        assert first > 0 and second == 0 and threads == 0, (m, runs)
        assert a == b and len(a) > 0
