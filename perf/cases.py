"""What the library's speed is measured on: filter chains over multichannel FP32 audio, through the Python entry points.

`listed()` are fixed cases, `draw()` makes more of the same ranges; `prepare()` builds what a program has in hand
before the call, `run()` is one pass, `work()` counts what a pass cannot do without, and `exact()` is the same result
in 64 bits from plain torch (the transfer function at the bins of one long transform, no code of this package)."""
import math

import numpy as np
import torch

from paper_2504_08624_gb300 import api
from paper_2504_08624_gb300 import workloads as W

FS = 48000.0


# ---------------------------------------------------------------------------
# the chains


def stages_of(case):
    """The stage list [("sos", rows) | ("fir", taps), ...] of a forward case."""
    d = case["design"]
    if d == "plain":  # low-pass cascade, then a high-pass FIR
        return [("sos", W.butter_sos(4, 1000.0, FS)), ("fir", W.fir_highpass(case["taps"], 100.0, FS))]
    if d == "eq":  # anti-alias low-pass, a peaking equaliser, then a linear-phase low-pass
        return [("sos", W.cheby1_sos(8, 0.5, 8000.0, FS)), ("sos", W.random_peaking_bank(case["peaks"], FS, 2)),
                ("fir", W.fir_lowpass(case["taps"], 16000.0, FS))]
    if d == "iir":  # one Butterworth low-pass
        return [("sos", W.butter_sos(case["order"], case["fc"], 44100.0))]
    if d == "iir4":  # the paper's chain of four IIR filters
        return W.table4_chain().stages
    if d == "fir":  # one linear-phase low-pass
        return [("fir", W.fir_lowpass(case["taps"], case["fc"], FS))]
    if d == "band":  # one Kaiser band-pass
        return [("fir", W.fir_bandpass(case["taps"], 300.0, 3400.0, FS, ("kaiser", 8.0)))]
    if d == "subsonic":  # rumble filter: high-pass with poles next to the unit circle
        return [("sos", W.butter_sos(case["order"], case["fc"], FS, "high"))]
    if d == "random":  # random stable sections and a low-pass FIR
        return W.random_chain(case["chain"])
    raise ValueError(d)


def sections_and_taps(stages):
    return sum(len(c) for k, c in stages if k == "sos"), [len(c) for k, c in stages if k == "fir"]


# ---------------------------------------------------------------------------
# the cases


def listed():
    return [
        # one mono sound effect of half a second through its own plan: a call is one short launch, latency is all
        {"name": "mono_half_second", "kind": "plan", "design": "random", "chain": 12, "signal": "uniform",
         "C": 1, "N": 24001, "pad": 0},
        # ten seconds of stereo through the one-shot call, as a script filters a file (no plan in the caller's hands)
        {"name": "stereo_ten_seconds", "kind": "call", "design": "plain", "taps": 101, "signal": "uniform",
         "C": 2, "N": 480000, "pad": 0},
        # a 33-tap FIR over 30 s of 5.1 sound: the shortest FIRs of the many-clip workload
        {"name": "short_fir_5p1", "kind": "call", "design": "fir", "taps": 33, "fc": 9000.0, "signal": "gauss",
         "C": 6, "N": 1440007, "pad": 0},
        # one cell of the paper's IIR timing grid: 12 channels x 180 s at 44.1 kHz, fourth-order Butterworth
        {"name": "iir_grid_12ch_180s", "kind": "call", "design": "iir", "order": 4, "fc": 1000.0, "signal": "gauss",
         "C": 12, "N": 7938000, "pad": 0},
        # the paper's chain of four IIR filters, 8 channels x 120 s at 44.1 kHz
        {"name": "iir_chain_8ch_120s", "kind": "plan", "design": "iir4", "signal": "gauss",
         "C": 8, "N": 5292000, "pad": 0},
        # a multitrack session: equaliser and 1025-tap low-pass over 64 channels x 60 s
        {"name": "multitrack_eq_64ch_60s", "kind": "plan", "design": "eq", "peaks": 4, "taps": 1025,
         "signal": "pink", "C": 64, "N": 2880000, "pad": 0},
        # a room response of 4097 taps over a ragged buffer: odd length, rows padded to an odd stride
        {"name": "room_response_ragged", "kind": "plan", "design": "band", "taps": 4097, "signal": "gauss",
         "C": 11, "N": 1000003, "pad": 38},
        # a 16384-tap band-pass over 128 channels x 4 Mi samples: the largest call
        {"name": "long_fir_128ch", "kind": "plan", "design": "band", "taps": 16384, "signal": "gauss",
         "C": 128, "N": 4194304, "pad": 0},
        # a rumble filter (10 Hz high-pass, poles beyond radius 0.999) over 8 channels x 60 s: exact long states
        {"name": "subsonic_8ch_60s", "kind": "plan", "design": "subsonic", "order": 2, "fc": 8.0, "signal": "pink",
         "C": 8, "N": 2880000, "pad": 0},
        # one MSE training step of six biquads and a 257-tap FIR, batch 256 x 65,536: outputs, loss and gradients
        {"name": "train_step_256x65536", "kind": "train", "sections": 6, "taps": 257, "C": 256, "N": 65536},
        # the same filters as a layer of a network under torch.autograd, batch 24 of one second
        {"name": "autograd_layer_24x48000", "kind": "layer", "sections": 6, "taps": 257, "C": 24, "N": 48000},
        # 120 clips of 0.5-30 s and 1-16 channels, each with its own chain, in one batched execution
        {"name": "batch_120_clips", "kind": "batch", "clips": 120, "seed": 5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same kinds of call, sizes spread over the logarithm, odd ones among them, at most 64 Mi
    channel-samples of a forward (of a training step 16 Mi)."""
    kind = rng.choice(["plan", "plan", "call", "train", "layer", "batch"])
    if kind == "batch":
        return {"kind": "batch", "clips": _log_int(rng, 6, 120), "seed": rng.randrange(1, 1000)}
    if kind in ("train", "layer"):
        C = _log_int(rng, 3, 256) if kind == "train" else _log_int(rng, 3, 48)
        return {"kind": kind, "sections": rng.randint(2, 6), "taps": 2 * _log_int(rng, 16, 128) + 1,
                "C": C, "N": _log_int(rng, 12000, 65536)}
    C = rng.choice([1, 2, 3, 6, 8, 11, 12, 16, 32, 64])
    N = _log_int(rng, 24000, min(8000000, 67108864 // C))
    case = {"kind": kind, "C": C, "N": N, "pad": rng.choice([0, 0, rng.randint(1, 64)]),
            "signal": rng.choice(["uniform", "gauss", "pink"])}
    d = rng.choice(["plain", "eq", "iir", "iir4", "fir", "band", "subsonic", "random"])
    case["design"] = d
    if d == "plain":
        case["taps"] = 2 * _log_int(rng, 16, 1024) + 1
    elif d == "eq":
        case["peaks"], case["taps"] = rng.randint(1, 6), 2 * _log_int(rng, 16, 1024) + 1
    elif d == "iir":
        case["order"], case["fc"] = rng.randint(2, 8), math.exp(rng.uniform(math.log(300.0), math.log(12000.0)))
    elif d == "fir":
        case["taps"], case["fc"] = 2 * _log_int(rng, 16, 1024) + 1, rng.uniform(2000.0, 20000.0)
    elif d == "band":
        case["taps"] = _log_int(rng, 1024, 16384)
        case["N"] = max(N, 100001)
    elif d == "subsonic":
        case["order"], case["fc"] = 2, rng.uniform(4.0, 9.0)
    elif d == "random":
        case["chain"] = rng.randrange(1, 100000)
    return case


# ---------------------------------------------------------------------------
# inputs


def _noise(C, N, signal, gen, pad=0):
    """[C x N] FP32 noise on the GPU, its rows N + pad apart."""
    x = torch.empty((C, N + pad), dtype=torch.float32, device="cuda")[:, :N]
    if signal == "uniform":
        x.uniform_(-1.0, 1.0, generator=gen)
    elif signal == "gauss":
        x.normal_(generator=gen)
    elif signal == "pink":  # 1/f power, RMS 0.1 per channel
        n = 1 << (N - 1).bit_length()
        shape = torch.arange(n // 2 + 1, device="cuda", dtype=torch.float32).clamp_(min=1.0).rsqrt_()
        shape[0] = 0.0
        for c in range(C):
            s = torch.fft.irfft(torch.fft.rfft(torch.randn(n, device="cuda", generator=gen)) * shape, n=n)[:N]
            x[c] = s * (0.1 / s.square().mean().sqrt())
    else:
        raise ValueError(signal)
    return x


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _train_inputs(case, seed):
    """Signal and target of a training case (the target: the signal, delayed and scaled, plus noise) and the
    parameters of its filters."""
    g = _gen(seed)
    x = _noise(case["C"], case["N"], "gauss", g)
    t = 0.5 * torch.roll(x, 3, dims=1) + 0.1 * _noise(case["C"], case["N"], "gauss", g)
    return x, t, W.differentiable_chain_params(41, case["sections"], case["taps"])


def _batch_clips(case):
    return W.batched_clips(case["clips"], case["seed"])


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("plan", "call"):
        stages = stages_of(case)
        x = _noise(case["C"], case["N"], case["signal"], _gen(seed), case["pad"])
        s = {"kind": kind, "x": x, "stages": stages}
        if kind == "plan":
            ld = case["N"] + case["pad"]
            s["plan"] = api.Plan(case["C"], case["N"], stages, ld=ld)
            s["plan"].workspace()
            s["y"] = torch.empty((case["C"], ld), dtype=torch.float32, device="cuda")[:, :case["N"]]
        return s
    if kind == "train":
        x, t, p = _train_inputs(case, seed)
        stages = [("sos", W.biquad_rows(p["rho"], p["phi"], p["b"])), ("fir", p["h"])]
        plan = api.Plan(case["C"], case["N"], stages, flags=api.N.TFX_PLAN_TRAINABLE)
        plan.train_workspace()
        return {"kind": kind, "plan": plan, "x": x, "t": t, "y": torch.empty_like(x), "g": torch.empty_like(x),
                "dx": torch.empty_like(x), "loss": torch.empty(1, dtype=torch.float64, device="cuda"),
                "dc": torch.empty(plan.coef_count, dtype=torch.float64, device="cuda"), "saved": plan.new_saved()}
    if kind == "layer":
        x, t, p = _train_inputs(case, seed)
        layer = api.LearnableBiquadChain(p["rho"], p["phi"], p["b"], p["h"]).cuda()
        return {"kind": kind, "layer": layer, "x": x.requires_grad_(True), "t": t}
    if kind == "batch":
        clips = _batch_clips(case)
        batch = api.Batch([(c.C, c.N, c.stages) for c in clips])
        batch.workspace()
        x = batch.empty()
        x.uniform_(-1.0, 1.0, generator=_gen(seed))
        return {"kind": kind, "batch": batch, "x": x, "y": torch.zeros_like(x)}
    raise ValueError(kind)


def run(state):
    kind = state["kind"]
    if kind == "plan":
        return {"y": state["plan"].execute(state["x"], state["y"])}
    if kind == "call":
        return {"y": api.chain(state["x"], state["stages"])}
    if kind == "train":
        s = state
        s["plan"].train_step_mse(s["x"], s["y"], s["t"], s["g"], s["loss"], s["dx"], s["dc"], s["saved"])
        return {"y": s["y"], "g": s["g"], "loss": s["loss"], "dx": s["dx"], "dcoef": s["dc"]}
    if kind == "layer":
        layer, x = state["layer"], state["x"]
        y = layer(x)
        loss = api.mse_loss(y, state["t"])
        grads = torch.autograd.grad(loss, [x, layer.rho, layer.phi, layer.b, layer.h])
        return {"y": y.detach(), "loss": loss.detach(), **dict(zip(("dx", "rho", "phi", "b", "h"), grads))}
    if kind == "batch":
        return {"y": state["batch"].execute(state["x"], state["y"])}
    raise ValueError(kind)


# ---------------------------------------------------------------------------
# what a pass cannot do without


def _filter_flops(S, taps):
    """Per channel-sample: 10 for a section; an FIR directly, or by transforms where those need less."""
    return 10.0 * S + sum(min(2.0 * L, 10.0 * math.log2(2.0 * L)) for L in taps)


def work(case):
    kind = case["kind"]
    if kind in ("plan", "call"):
        n = float(case["C"]) * case["N"]
        return {"bytes": 8.0 * n, "flops": n * _filter_flops(*sections_and_taps(stages_of(case)))}
    if kind in ("train", "layer"):  # in: signal, target; out: y, dx (and the step's g); forward, dx, correlation
        n = float(case["C"]) * case["N"]
        return {"bytes": (20.0 if kind == "train" else 16.0) * n,
                "flops": 3.0 * n * _filter_flops(case["sections"], [case["taps"]])}
    total = {"bytes": 0.0, "flops": 0.0}
    for c in _batch_clips(case):
        n = float(c.C) * c.N
        total["bytes"] += 8.0 * n
        total["flops"] += n * _filter_flops(*sections_and_taps(c.stages))
    return total


# ---------------------------------------------------------------------------
# the same in 64 bits


def _tail(stages):
    """Samples after which the chain's response is below 1e-17 of its start (pole radius r: r^n), plus its taps."""
    n = 64
    for k, c in stages:
        if k == "fir":
            n += len(c)
        else:
            for row in np.asarray(c, dtype=np.float64):
                r = float(np.max(np.abs(np.roots(row[3:])))) if np.any(row[4:] != 0.0) else 0.0
                if r > 0.0:
                    n = n + int(math.ceil(45.0 / -math.log(min(r, 0.99999)))) + 1
    return n


def _transfer(coefs, n):
    """H at the rfft bins of an n-point transform, complex128 torch; differentiable in the coefficients."""
    w = torch.arange(n // 2 + 1, dtype=torch.float64, device="cuda") * (-2.0 * math.pi / n)
    z = torch.polar(torch.ones_like(w), w)
    z2 = z * z
    h = torch.ones_like(z)
    for kind, c in coefs:
        if kind == "fir":
            h = h * torch.fft.rfft(c, n=n)
        else:
            for r in c:
                h = h * (r[0] + r[1] * z + r[2] * z2) / (r[3] + r[4] * z + r[5] * z2)
    return h


def _coefs64(stages):
    return [(k, torch.as_tensor(np.asarray(c), dtype=torch.float64, device="cuda")) for k, c in stages]


def _length(N, stages):
    n = N + _tail(stages)
    return 1 << (n - 1).bit_length()


def _filter64(x, stages, reverse=False):
    C, N = x.shape
    n = _length(N, stages)
    h = _transfer(_coefs64(stages), n)
    y = torch.empty((C, N), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 26) // n)
    for c in range(0, C, step):
        u = x[c:c + step].double()
        u = u.flip(1) if reverse else u
        v = torch.fft.irfft(torch.fft.rfft(u, n=n) * h, n=n)[:, :N]
        y[c:c + step] = v.flip(1) if reverse else v
    return y


def _gradients64(x, t, stages, params, coefs):
    """y, loss, dL/dy, dL/dx and dL/d(params) of the MSE step; `coefs`: the stages as torch functions of `params`."""
    C, N = x.shape
    y = _filter64(x, stages)
    d = y - t.double()
    g = d * (2.0 / (C * N))
    n = _length(N, stages)
    cross = torch.zeros(n // 2 + 1, dtype=torch.complex128, device="cuda")
    step = max(1, (1 << 25) // n)
    for c in range(0, C, step):
        X = torch.fft.rfft(x[c:c + step].double(), n=n)
        cross += (X * torch.fft.rfft(g[c:c + step], n=n).conj()).sum(0)
    weight = torch.full((n // 2 + 1,), 2.0 / n, dtype=torch.float64, device="cuda")
    weight[0] = weight[-1] = 1.0 / n
    inner = ((_transfer(coefs, n) * cross).real * weight).sum()  # sum g y
    return y, d.square().mean(), g, _filter64(g, stages, reverse=True), torch.autograd.grad(inner, params)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("plan", "call"):
        x = _noise(case["C"], case["N"], case["signal"], _gen(seed), case["pad"])
        return {"y": _filter64(x, stages_of(case))}
    if kind in ("train", "layer"):
        x, t, p = _train_inputs(case, seed)
        stages = [("sos", W.biquad_rows(p["rho"], p["phi"], p["b"])), ("fir", p["h"])]
        if kind == "train":
            rows, taps = (c.clone().requires_grad_(True) for _, c in _coefs64(stages))
            y, loss, g, dx, (dr, dh) = _gradients64(x, t, stages, [rows, taps], [("sos", rows), ("fir", taps)])
            return {"y": y, "g": g, "loss": loss.reshape(1), "dx": dx, "dcoef": torch.cat([dr.reshape(-1), dh])}
        rho, phi, b, h = (torch.as_tensor(p[k], dtype=torch.float64, device="cuda").requires_grad_(True)
                          for k in ("rho", "phi", "b", "h"))
        r = 0.5 + 0.49 * torch.sigmoid(rho)
        th = math.pi * torch.sigmoid(phi)
        rows = torch.cat([b, torch.stack([torch.ones_like(r), -2.0 * r * torch.cos(th), r * r], 1)], 1)
        y, loss, _, dx, grads = _gradients64(x, t, stages, [rho, phi, b, h], [("sos", rows), ("fir", h)])
        return {"y": y, "loss": loss, "dx": dx, **dict(zip(("rho", "phi", "b", "h"), grads))}
    clips = _batch_clips(case)  # packed one after the other, each [C x N]
    x = torch.empty(sum(c.C * c.N for c in clips), dtype=torch.float32, device="cuda")
    x.uniform_(-1.0, 1.0, generator=_gen(seed))
    y, o = torch.empty(x.shape, dtype=torch.float64, device="cuda"), 0
    for c in clips:
        n = c.C * c.N
        y[o:o + n] = _filter64(x[o:o + n].view(c.C, c.N), c.stages).reshape(-1)
        o += n
    return {"y": y}
