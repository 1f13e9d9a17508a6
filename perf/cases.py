"""The work a spectrometer user has the library do, as a list of timed cases.

Three kinds of case, each through the public Python entry points:
  "spectra"  Spectrometer: feed packed IF streams, close the integration (autos, crosses, Stokes)
  "leakage"  Adjoint.run / leakage_loss: leakage-calibration loss and its gradients
  "tensor"   TensorCoreSpectrometer: the tensor-core precision variant
`listed` names one case per use, `draw` gives others of the same ranges.  `exact` restates each
in plain torch in 64 bits.
"""
import math

import numpy as np
import torch

from paper_1412_1256_gb300 import polaris

# fields of a spectra case and their usual values
SPECTRA = {
    "kind": "spectra", "n_if": 4, "bits": 2, "log2n": 17, "segments": 61,
    "one_pair": False,   # only IFs (0, 1) are correlated (the others give autos alone)
    "window": "rect",    # rect, hann or custom (Blackman taps handed over as an array)
    "overlap": False,    # 50% overlap (hop = N/2), in the steady state of a running stream
    "fp64": False,       # FP64 integration accumulators
    "circular": False,   # circular feeds, parallactic angle and per-IF gains
    "chunks": 1,         # the stream arrives in this many uneven pieces
    "host": False,       # host buffers in and out (pinned) instead of device tensors
    "stats": False,      # code statistics on, read and reset with every integration
    "handles": 0,        # > 0: that many handles, each on a stream of its own, phase 1 capped at
    "steps": 1,          #   one CTA per SM, take `steps` consecutive integrations in turn
}


def spectra(name, **kw):
    return {"name": name, **SPECTRA, **kw}


def listed():
    return [
        # the smallest call: a quick look at two int8 IFs, 1024 points, 64 segments (launches and latency)
        spectra("quick_look_1k", n_if=2, bits=8, log2n=10, segments=64, window="hann"),
        # a stream that arrives in uneven pieces (samples carried from feed to feed), an IF without a
        # partner, an own window
        spectra("ragged_feeds_4k", n_if=3, bits=4, log2n=12, segments=601, one_pair=True, window="custom", chunks=7),
        # few wide channels over many IFs of 1-bit samples
        spectra("wide_channels_2k", n_if=8, bits=1, log2n=11, segments=2441),
        # 1 s of four 16-Msps 8-bit IFs, Hann window with 50% overlap (no loss of sensitivity)
        spectra("overlap_16k", n_if=4, bits=8, log2n=14, segments=1953, window="hann", overlap=True),
        # the paper's 1-s integration: four IFs, 2-bit, 131072-point segments, device-resident
        spectra("paper_1s"),
        # the same second as a telescope's back end has it: from pinned host buffers, spectra back
        # to the host, with the bit distribution for the total power; 4-bit samples
        spectra("real_time_host_1s", bits=4, host=True, stats=True),
        # a recording played back as fast as it goes: three handles on three streams, six seconds
        spectra("playback_6s", handles=3, steps=6),
        # the finest channels: 2^20 points, int8, Hann, circular feeds with gains, 1 s at 16 Msps
        spectra("fine_channels_1m", n_if=2, bits=8, log2n=20, segments=15, window="hann", circular=True),
        # a long integration of a strong line: 10 s at 16 Msps, 2^18 points, FP64 accumulators
        spectra("long_10s", n_if=2, bits=8, log2n=18, segments=610, window="hann", fp64=True),
        # one step of the leakage calibration: Stokes, loss and every gradient, 16384 x 256 segments
        {"name": "calibration_16k", "kind": "leakage", "bits": 8, "log2n": 14, "segments": 256, "autograd": False},
        # a small calibration inside a torch optimiser: the loss and its backward pass
        {"name": "calibration_autograd_1k", "kind": "leakage", "bits": 2, "log2n": 10, "segments": 61, "autograd": True},
        # the tensor-core variant's spectra of one second at 2^18 points
        {"name": "tensor_core_256k", "kind": "tensor", "bits": 8, "log2n": 18, "segments": 61, "window": "hann",
         "precision": "fp16x3"},
    ]


def log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(("spectra",) * 6 + ("leakage", "leakage", "tensor"))
    bits = rng.choice((1, 2, 4, 8))
    if kind == "leakage":
        log2n = rng.randint(6, 14)
        samples = log_uniform(rng, 2.0 ** 15, 2.0 ** 22)
        return {"kind": kind, "bits": bits, "log2n": log2n, "segments": max(1, int(samples / 2 ** log2n)),
                "autograd": rng.random() < 0.5}
    if kind == "tensor":
        log2n = rng.choice((12, 18))
        samples = log_uniform(rng, 2.0 ** 18, 2.0 ** 25)
        return {"kind": kind, "bits": bits, "log2n": log2n, "segments": max(1, int(samples / 2 ** log2n)),
                "window": rng.choice(("rect", "hann", "custom")), "precision": rng.choice(("fp16x3", "bf16x3", "bf16"))}
    c = dict(SPECTRA)
    c["bits"], c["log2n"] = bits, rng.randint(8, 20)
    c["n_if"] = rng.choice((1, 2, 2, 3, 4, 4, 5, 8))
    samples = log_uniform(rng, 2.0 ** 16, 2.0 ** 27) / c["n_if"]
    c["segments"] = max(1, int(samples / 2 ** c["log2n"]))
    c["one_pair"] = c["n_if"] > 1 and rng.random() < 0.2
    c["window"] = rng.choice(("rect", "hann", "custom"))
    c["overlap"] = rng.random() < 0.25
    c["fp64"] = rng.random() < 0.25
    c["circular"] = rng.random() < 0.3
    way = rng.choice(("whole", "whole", "chunks", "host", "handles"))
    if way == "chunks":
        c["chunks"] = rng.randint(2, 9)
    elif way == "host":
        c["host"] = True
        c["segments"] = max(1, c["segments"] // 4)
    elif way == "handles":
        c["handles"], c["steps"] = 3, 4
        c["segments"] = max(1, c["segments"] // 4)
        c["overlap"] = False
    c["stats"] = way != "handles" and rng.random() < 0.25
    return c


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def pair_list(case):
    n = case["n_if"]
    if case["one_pair"]:
        return [(0, 1)]
    return [(i, i + n // 2) for i in range(n // 2)] if n % 2 == 0 else []


def taps_of(window, n):
    """Window taps in 64 bits, from the float32 values that the library is given or makes."""
    t = torch.arange(n, dtype=torch.float64)
    if window == "rect":
        return torch.ones(n, dtype=torch.float64)
    if window == "hann":
        return (0.5 - 0.5 * torch.cos(2 * math.pi * t / n)).float().double()
    a = 2 * math.pi * t / n
    return (0.42 - 0.5 * torch.cos(a) + 0.08 * torch.cos(2 * a)).float().double()


def window_arg(window, n):
    return window if window in ("rect", "hann") else taps_of(window, n).float().numpy()


def sampled(n_if, n_samples, bits, n_fft, seed):
    """Packed words [n_if, n_samples * bits / 32] (int32, on the GPU): Gaussian noise and a weak
    line common to all IFs (a quarter turn later in the second half of them), as a b-bit sampler
    quantises it."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    out = torch.empty((n_if, n_samples * bits // 32), dtype=torch.int32, device="cuda")
    spw, step = 32 // bits, 1 << 24
    freq = 0.25 * n_fft * (1 + 0.3 * torch.rand(1, generator=gen, device="cuda", dtype=torch.float64)) / n_fft
    for i in range(n_if):
        lag = 0.25 if i >= (n_if + 1) // 2 else 0.0
        for s0 in range(0, n_samples, step):
            n = min(step, n_samples - s0)
            turn = torch.arange(s0, s0 + n, device="cuda", dtype=torch.float64) * freq - lag
            v = torch.randn(n, generator=gen, device="cuda") + 0.3 * torch.cos(2 * math.pi * (turn - turn.floor()).float())
            if bits == 8:
                words = (20.0 * v).round_().clamp_(-128, 127).to(torch.int8).view(torch.int32)
            else:
                if bits == 1:
                    code = (v >= 0).to(torch.int32)
                elif bits == 2:
                    code = torch.bucketize(v, torch.tensor([-0.98, 0.0, 0.98], device="cuda"), right=True).to(torch.int32)
                else:
                    code = ((2.0 * v).floor() + 8).clamp_(0, 15).to(torch.int32)
                shifts = torch.arange(spw, dtype=torch.int32, device="cuda") * bits
                words = (code.view(-1, spw) << shifts).sum(dim=1).to(torch.int32)
            out[i, s0 // spw:(s0 + n) // spw] = words
    return out


def levels(words, bits):
    """Float64 levels of packed words (one stream)."""
    if bits == 8:
        return words.view(torch.int8).double()
    shifts = torch.arange(32 // bits, dtype=torch.int32, device=words.device) * bits
    return (2 * ((words.unsqueeze(1) >> shifts) & ((1 << bits) - 1)) - ((1 << bits) - 1)).reshape(-1).double()


def pieces(case):
    """Sample counts of the pieces in which the stream of one pass arrives."""
    spw = 32 // case["bits"]
    hop = 2 ** case["log2n"] // (2 if case["overlap"] else 1)
    words = case["segments"] * hop // spw
    k = min(case["chunks"], words)
    cuts = np.sort(np.random.RandomState(7).choice(np.arange(1, words), k - 1, replace=False)) if k > 1 else []
    edges = [0, *[int(c) for c in cuts], words]
    return [(b - a) * spw for a, b in zip(edges, edges[1:])]


def stokes_args(case):
    if not case["circular"]:
        return {}
    gains = [(complex(1.1, 0.2 * p), complex(0.9, -0.3)) for p in range(len(pair_list(case)))]
    return {"feed": polaris.FEED_CIRCULAR, "psi": 0.4, "gains": gains or None}


def leakage_inputs(case, seed):
    n, nb = 2 ** case["log2n"], 2 ** case["log2n"] // 2 + 1
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def rnd(*shape):
        return torch.randn(*shape, generator=gen, device="cuda")

    window = taps_of("hann", n).float().cuda()
    gains = torch.tensor([1.05, 0.1, 0.9, -0.15], device="cuda") + 0.02 * rnd(4)
    leak = 0.03 * rnd(2, nb, 2)
    # the calibrator: its power per bin, with a line of known polarisation
    power = {8: 400.0, 4: 16.0, 2: 3.5, 1: 1.0}[case["bits"]] * case["segments"] * float((window * window).sum())
    k = torch.arange(nb, device="cuda", dtype=torch.float32)
    line = torch.exp(-0.5 * ((k - 0.3 * nb) / (0.02 * nb)) ** 2)
    target = power * torch.stack([1 + line, 0.3 * line, -0.2 * line, 0.1 * line])
    return window, gains, leak, target


# ---------------------------------------------------------------------------------------------
# a user's program: what it keeps, and one pass
# ---------------------------------------------------------------------------------------------
def prepare(case, seed):
    n_fft, bits, segs = 2 ** case["log2n"], case["bits"], case["segments"]
    if case["kind"] == "leakage":
        window, gains, leak, target = leakage_inputs(case, seed)
        words = sampled(2, segs * n_fft, bits, n_fft, seed + 1)
        if case["autograd"]:
            for t in (window, gains, leak):
                t.requires_grad_(True)
        return {"case": case, "adj": polaris.Adjoint(n_fft, bits), "packed": [words[0], words[1]], "n": segs * n_fft,
                "window": window, "gains": gains, "leak": leak, "target": target}
    if case["kind"] == "tensor":
        words = sampled(2, segs * n_fft, bits, n_fft, seed)
        tc = polaris.TensorCoreSpectrometer(bits, n_fft, case["precision"], window_arg(case["window"], n_fft))
        return {"case": case, "tc": tc, "packed": [words[0], words[1]], "n": segs * n_fft}

    n_if, pairs = case["n_if"], pair_list(case)
    hop = n_fft // 2 if case["overlap"] else n_fft
    n, nb = segs * hop, n_fft // 2 + 1

    def handle():
        return polaris.Spectrometer(n_if, bits, n_fft, hop=hop, window=window_arg(case["window"], n_fft),
                                    pairs=pairs if case["one_pair"] else None, accum_fp64=case["fp64"],
                                    code_stats=case["stats"])

    def buffers(**kw):
        return {"autos": torch.empty((n_if, nb), **kw), "cross": torch.empty((len(pairs), nb, 2), **kw) if pairs else None,
                "stokes": torch.empty((len(pairs), 4, nb), **kw) if pairs else None}

    state = {"case": case, "stokes_args": stokes_args(case)}
    if case["handles"]:
        state["words"] = [sampled(n_if, n, bits, n_fft, seed + k) for k in range(case["steps"])]
        state["packed"] = [[w[i] for i in range(n_if)] for w in state["words"]]
        state["handles"] = [handle() for _ in range(case["handles"])]
        for h in state["handles"]:
            h.set_launch_caps(1, 0)
        state["streams"] = [torch.cuda.Stream() for _ in range(case["handles"])]
        state["out"] = [buffers(device="cuda") for _ in range(case["steps"])]
        state["n"] = n
        return state
    words = sampled(n_if, n, bits, n_fft, seed)
    sp = state["sp"] = handle()
    if case["overlap"]:
        # a running stream: the handle carries the last half segment from pass to pass
        tail = words[:, -(n_fft - hop) * bits // 32:] if n >= n_fft - hop else words
        tail = tail.contiguous()
        sp.feed([tail[i] for i in range(n_if)], n_fft - hop)
    if case["host"]:
        words = words.cpu().pin_memory()
        out = {k: None if t is None else t.pin_memory() for k, t in buffers().items()}
        state["out"] = {k: t.numpy() for k, t in out.items() if t is not None}
        state["keep"] = out
        rows = words.numpy().view(np.uint32)
    else:
        state["out"] = buffers(device="cuda")
        rows = words
    state["words"], state["feeds"], at = words, [], 0
    for m in pieces(case):
        w = m * bits // 32
        state["feeds"].append(([rows[i, at:at + w] for i in range(n_if)], m))
        at += w
    torch.cuda.synchronize()
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "leakage":
        if not case["autograd"]:
            return state["adj"].run(state["packed"], state["n"], state["window"], state["gains"], state["leak"],
                                    state["target"], grads=True, stream=torch.cuda.current_stream())
        params = (state["window"], state["gains"], state["leak"])
        loss = polaris.leakage_loss(state["adj"], state["packed"], state["n"], *params, state["target"])
        return {"loss": loss.detach(), "grads": torch.autograd.grad(loss, params)}
    if case["kind"] == "tensor":
        stream = torch.cuda.current_stream()
        state["tc"].feed(state["packed"], state["n"], stream=stream)
        got = state["tc"].integrate(stream=stream)
        return {"autos": got["autos"], "cross": got["cross"], "stokes": got["stokes"]}
    if case["handles"]:
        here = torch.cuda.current_stream()
        for s in state["streams"]:
            s.wait_stream(here)
        for k, (packed, out) in enumerate(zip(state["packed"], state["out"])):
            h, s = state["handles"][k % case["handles"]], state["streams"][k % case["handles"]]
            h.feed(packed, state["n"], stream=s)
            h.integrate_device(out["autos"], out["cross"], out["stokes"], stream=s, **state["stokes_args"])
        for s in state["streams"]:
            here.wait_stream(s)
        return state["out"]
    sp, out = state["sp"], state["out"]
    if case["host"]:
        for packed, m in state["feeds"]:
            sp.feed(packed, m)
        sp.integrate(out=out, **state["stokes_args"])
    else:
        stream = torch.cuda.current_stream()
        for packed, m in state["feeds"]:
            sp.feed(packed, m, stream=stream)
        sp.integrate_device(out["autos"], out["cross"], out["stokes"], stream=stream, **state["stokes_args"])
    if case["stats"]:
        return {"spectra": out, "codes": sp.code_histogram(reset=True).view(np.int64)}
    return {"spectra": out}


def work(case):
    n, segs, bits = 2 ** case["log2n"], case["segments"], case["bits"]
    nb, fft = n // 2 + 1, 2.5 * n * case["log2n"]  # one real transform
    if case["kind"] == "leakage":
        # inputs, window, target and parameters in; Stokes and gradients out.  Three transforms of
        # each segment pair at most are needed: forward, adjoint back
        words = 2 * segs * n * bits / 8
        return {"bytes": words + 4 * (2 * n + 4 * nb + 4 * nb + 8 * nb + 8), "flops": segs * (2 * 2 * fft + 40 * nb + 8 * n)}
    if case["kind"] == "tensor":
        return {"bytes": 2 * segs * n * bits / 8 + 8 * 8 * nb, "flops": segs * (2 * fft + 16 * nb + 2 * n)}
    hop = n // 2 if case["overlap"] else n
    pairs, steps = len(pair_list(case)), case["steps"]
    out = 4 * nb * (case["n_if"] + 6 * pairs)
    taps = 4 * n if case["window"] != "rect" else 0
    win = n if case["window"] != "rect" else 0
    flops = segs * (case["n_if"] * (fft + win + 4 * nb) + 8 * nb * pairs)
    return {"bytes": steps * (case["n_if"] * segs * hop * bits / 8 + out + taps), "flops": steps * flops}


# ---------------------------------------------------------------------------------------------
# the same results in plain torch, 64 bits
# ---------------------------------------------------------------------------------------------
def exact_spectra(words, case, window):
    """autos, cross of one integration: words [n_if, words], segments at the case's hop (cyclic
    with overlap: the handle carries the previous pass's last half segment)."""
    n, segs, bits, pairs = 2 ** case["log2n"], case["segments"], case["bits"], pair_list(case)
    hop = n // 2 if case.get("overlap") else n
    nb = n // 2 + 1
    autos = torch.zeros((case["n_if"], nb), dtype=torch.float64, device="cuda")
    cross = torch.zeros((len(pairs), nb), dtype=torch.complex128, device="cuda")
    wph = hop * bits // 32
    if case.get("overlap"):
        words = torch.cat([words[:, -wph:], words], dim=1)
    step = max(1, (1 << 23) // n)
    for s0 in range(0, segs, step):
        k = min(step, segs - s0)
        spec = []
        for i in range(case["n_if"]):
            x = levels(words[i, s0 * wph:(s0 + k - 1) * wph + n * bits // 32], bits).unfold(0, n, hop)
            spec.append(torch.fft.rfft(x * window, dim=1))
            autos[i] += (spec[i].real ** 2 + spec[i].imag ** 2).sum(dim=0)
        for p, (a, b) in enumerate(pairs):
            cross[p] += (spec[a] * spec[b].conj()).sum(dim=0)
        del spec
    return autos, cross


def exact_stokes(case, autos, cross):
    args = stokes_args(case) if case["kind"] == "spectra" else {}
    rows = []
    for p, (a, b) in enumerate(pair_list(case)):
        ga, gb = args["gains"][p] if args.get("gains") else (1.0, 1.0)
        ga, gb = complex(np.complex64(ga)), complex(np.complex64(gb))
        x, y = autos[a] / abs(ga) ** 2, autos[b] / abs(gb) ** 2
        c = cross[p] / (ga * gb.conjugate())
        c2, s2 = math.cos(2 * args.get("psi", 0.0)), math.sin(2 * args.get("psi", 0.0))
        if args.get("feed", polaris.FEED_LINEAR) == polaris.FEED_CIRCULAR:
            rows.append(torch.stack([(x + y) / 2, c2 * c.real - s2 * c.imag, s2 * c.real + c2 * c.imag, (x - y) / 2]))
        else:
            rows.append(torch.stack([(x + y) / 2, (c2 * (x - y) - s2 * 2 * c.real) / 2,
                                     (s2 * (x - y) + c2 * 2 * c.real) / 2, c.imag]))
    return torch.stack(rows) if rows else None


def exact_leakage(case, seed):
    window, gains, leak, target = (t.double() for t in leakage_inputs(case, seed))
    n, segs = 2 ** case["log2n"], case["segments"]
    words = sampled(2, segs * n, case["bits"], n, seed + 1)
    for t in (window, gains, leak):
        t.requires_grad_(True)
    x, y = (torch.fft.rfft(levels(words[i], case["bits"]).view(segs, n) * window, dim=1) for i in (0, 1))
    g_r, g_l = torch.complex(gains[0], gains[1]), torch.complex(gains[2], gains[3])
    d = torch.view_as_complex(leak)
    r, l = g_r * (x + d[0] * y), g_l * (y + d[1] * x)
    rr, ll = (r.real ** 2 + r.imag ** 2).sum(dim=0), (l.real ** 2 + l.imag ** 2).sum(dim=0)
    rl = (r * l.conj()).sum(dim=0)
    stokes = torch.stack([(rr + ll) / 2, rl.real, rl.imag, (rr - ll) / 2])
    loss = ((stokes - target) ** 2).sum()
    grads = torch.autograd.grad(loss, (window, gains, leak))
    if case["autograd"]:
        return {"loss": loss.detach(), "grads": grads}
    return {"stokes": stokes.detach(), "loss": loss.detach().reshape(1), "grad_window": grads[0], "grad_gains": grads[1],
            "grad_leak": grads[2]}


def exact(case, seed):
    if case["kind"] == "leakage":
        return exact_leakage(case, seed)
    n, segs, bits = 2 ** case["log2n"], case["segments"], case["bits"]
    window = taps_of(case["window"], n).cuda()
    if case["kind"] == "tensor":
        one = {"kind": "tensor", "n_if": 2, "one_pair": False, "log2n": case["log2n"], "bits": bits, "segments": segs}
        autos, cross = exact_spectra(sampled(2, segs * n, bits, n, seed), one, window)
        return {"autos": autos, "cross": cross[0], "stokes": exact_stokes(one, autos, cross)[0]}
    hop = n // 2 if case["overlap"] else n
    got = []
    for k in range(case["steps"]):
        words = sampled(case["n_if"], segs * hop, bits, n, seed + k)
        autos, cross = exact_spectra(words, case, window)
        pairs = bool(pair_list(case))
        got.append({"autos": autos, "cross": torch.view_as_real(cross) if pairs else None,
                    "stokes": exact_stokes(case, autos, cross) if pairs else None})
    if case["handles"]:
        return got
    if not case["host"]:
        out = {"spectra": got[0]}
    else:
        out = {"spectra": {k: v for k, v in got[0].items() if v is not None}}
    if case["stats"]:
        out["codes"] = None
    return out
