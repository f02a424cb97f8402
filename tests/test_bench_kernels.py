"""The kernels that bench.py names: what each kind of unit launches, every name
a kernel of the sources, the transform flop count of a real block, and the
traffic records' kernels found in the files that they were taken from."""
import glob
import json
import os
import re

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _kernels(paths):
    names = set()
    for p in paths:
        with open(p) as f:
            names |= set(re.findall(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s+)?(\w+)\(", f.read()))
    return names


CSRC = _kernels(glob.glob(os.path.join(ROOT, "paper_2504_08624_gb300", "csrc", "*.cu*")))


def test_launched_kernels_per_route():
    f = bench.launched_kernels
    assert f({"kind": "chain_fft", "M": 16384, "B": 11154}) == "k_fir_rfft"
    assert f({"kind": "fir_fft", "L": 65, "M": 1024, "B": 960, "P": 0}) == "k_fir_rfft"
    assert f({"kind": "fir_fft", "L": 16384, "M": 16384, "B": 8192, "P": 2}) == "k_fir_fft_spec+k_fir_fft_conv"
    assert f({"kind": "fir", "L": 33}) == "k_fir_direct" and f({"kind": "fir", "L": 64}) == "k_unit"
    assert f({"kind": "cascade", "scan": "phase"}) == "k_sos_phase+k_carry_scan"
    assert f({"kind": "cascade", "scan": "warp"}) == "k_sos_warp" and f({"kind": "cascade", "scan": "tc"}) == "k_sos_tc"
    assert f({"kind": "fused", "S": 2, "L": 31}) == "k_unit"
    for name in "k_fir_rfft+k_fir_fft_spec+k_fir_fft_conv+k_fir_direct+k_sos_phase+k_carry_scan+k_sos_warp+k_unit".split("+"):
        assert name in CSRC, name


def test_names_in_the_bench_are_kernels():
    with open(os.path.join(ROOT, "bench.py")) as f:
        used = set(re.findall(r"\bk_(?:fir|sos|unit|chain|xcorr|spectral|carry)\w*", f.read()))
    assert "k_fir_rfft" in used and "k_fir_rfft_batched" in used
    assert used - {"k_fir_fft"} <= CSRC, used - CSRC  # (k_fir_fft: the FFT route's family)


def test_flops_of_a_real_block():
    # M = 4096 samples, 2048 points: two transforms of 10 levels of 5 flop per
    # point and the product, per 3072 outputs
    got = bench.fft_flops_per_output({"M": 4096, "B": 3072, "P": 0})
    assert abs(got - 2048 * (2 * 5 * 10 + 14) / 3072) < 1e-9


def test_traffic_records_name_kernels_of_their_sources():
    with open(os.path.join(ROOT, "profiles", "traffic.json")) as f:
        rec = json.load(f)
    for kernels, by_workload in rec.items():
        for e in by_workload.values():
            src = e["source"] if isinstance(e["source"], list) else [e["source"]]
            found = _kernels([os.path.join(ROOT, s) for s in src])
            for k in kernels.split("+"):
                assert k in found, (k, src)
