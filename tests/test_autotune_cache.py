"""The batch autotuner's cache and candidates, with the timing replaced (no
GPU): winners timed with another library build are not taken, every size that
the cost model may choose is a candidate, and a bucket that the cost model
serves best is left to it."""
import json
import types

import pytest

autotune = pytest.importorskip("paper_2504_08624_gb300.autotune")

CLIPS = [(2, 90000, [])] * 3


@pytest.fixture
def tuned(tmp_path, monkeypatch):
    lib = tmp_path / "lib.so"
    lib.write_bytes(b"one build")
    taps = [300]

    class Batch:
        def __init__(self, clips, **kw):
            pass

        def clip_info(self, i):
            return True, taps[0], 12

        def close(self):
            pass

    times = {}
    calls = []

    def time_clips(clips, reps, fft_m):
        (m,) = fft_m.values()
        calls.append(m)
        return times.get(m, 5.0)

    monkeypatch.setattr(autotune.api, "Batch", Batch)
    monkeypatch.setattr(autotune, "_time_clips", time_clips)
    monkeypatch.setattr(autotune, "_native", types.SimpleNamespace(LIB_PATH=str(lib)), raising=False)

    def run(length, best, build=None):
        if build:
            lib.write_bytes(build)
            getattr(autotune, "_build_tag", run.tag).cache_clear()
        taps[0] = length
        times.clear()
        times[best] = 1.0
        calls.clear()
        r = autotune.tune_batch(CLIPS, cache_path=str(tmp_path / "cache.json"))
        return r, list(calls)

    run.cache = tmp_path / "cache.json"
    run.tag = types.SimpleNamespace(cache_clear=lambda: None)
    return run


def test_winners_of_another_build_are_timed_again(tuned):
    tuned.cache.write_text(json.dumps({"fftm:L8": 11}))  # as kernels of earlier builds left it
    r, calls = tuned(300, best=12)
    assert r["fft_m"] == {8: 12} and calls and not r["cached"]
    r, calls = tuned(300, best=13)
    assert r["fft_m"] == {8: 12} and not calls and r["cached"]
    r, calls = tuned(300, best=13, build=b"another build")
    assert r["fft_m"] == {8: 13} and calls and not r["cached"]
    assert json.loads(tuned.cache.read_text())["fftm:L8"] == 11  # (nobody else's entry is touched)


def test_every_size_that_holds_the_response(tuned):
    for length, sizes in ((300, [0, 10, 11, 12, 13, 14, 15]), (9000, [0, 14, 15]), (12289, [0, 14, 15])):
        r, calls = tuned(length, best=15, build=b"%d" % length)
        assert calls == sizes and r["fft_m"] == {length.bit_length() - 1: 15}
    r, calls = tuned(20000, best=15, build=b"last")  # one size only: nothing to choose
    assert not calls and r["fft_m"] == {}


def test_the_cost_models_choice_may_win(tuned):
    r, calls = tuned(300, best=0)
    assert r["fft_m"] == {} and not r["cached"]
    r, calls = tuned(300, best=14)
    assert r["fft_m"] == {} and r["cached"] and not calls
