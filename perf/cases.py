"""Performance cases of the channelizer: what a user's program has it do.

Each case is one integration: the accumulator is cleared, a block of int8
voltages is channelized into it through a public entry point, and the
accumulated spectra are the output (float4 XX, YY, Re XY*, Im XY* per channel
dual-pol, float XX single-pol).

Entry points (the "entry" of a case):
  execute  Plan.execute on device-resident input (also with sub-bands)
  host     Plan.execute_host: pinned host input, copies overlapped with compute
  batch    Batch.execute: several banks in one graph launch
"""
from __future__ import annotations

import math

import torch

from paper_1411_0436_gb300 import vspec, workloads

DEV = "cuda:0"

# The batched multi-beam workload: (nchan, spectra), PFB and direct alternating.
BEAMS = [(b.nchan, b.nspectra) for b in workloads.CONFIGS["c5"]]


def _case(name, nchan, nspectra, mode="pfb", taps=8, npol=2, window="hann", nsub=1, entry="execute", signal="tones"):
    c = {"nchan": nchan, "nspectra": nspectra, "mode": mode, "taps": taps, "npol": npol, "window": window,
         "nsub": nsub, "entry": entry, "signal": signal}
    return dict(name=name, **c) if name else c


def listed():
    return [
        # a single-polarisation receiver, the smallest mode, a short dump: latency
        _case("pfb_1024_1pol_s64", 1024, 64, npol=1),
        # a capture loop's block at the narrowest VEGAS mode: a few spectra per call
        _case("pfb_4096_s10", 4096, 10),
        # few channels, a long integration (pulsar or transient work)
        _case("pfb_1024_s2048", 1024, 2048),
        # the eight-sub-band mode: 16 FFTs in parallel over interleaved input
        _case("subbands_8x4096_s501", 4096, 501, nsub=8),
        # a sharper filter than the default: 12 taps, Hamming window, ragged length
        _case("pfb12_16384_s777", 16384, 777, taps=12, window="hamming"),
        # the common single-sub-band dump
        _case("pfb_32768_s1000", 32768, 1000),
        # a single-polarisation receiver with many channels
        _case("pfb_65536_1pol_s301", 65536, 301, npol=1),
        # the paper's benchmark from host memory: copies in both directions included
        _case("host_pfb_65536_s1000", 65536, 1000, entry="host"),
        # no pre-filter, the finest VEGAS resolution
        _case("direct_524288_s256", 524288, 256, mode="direct", taps=1, window="rect", signal="noise"),
        # the longest transform the paper benchmarks, with the pre-filter
        _case("pfb_1048576_s100", 1048576, 100),
        # eight beams of mixed sizes in one graph launch
        _case("beams_8", 0, 0, mode="mixed", entry="batch", signal="noise"),
        # a long integration on a weak, narrow line
        _case("pfb_131072_s4096", 131072, 4096, signal="line"),
    ]


def draw(rng):
    """Another case of the same ranges: 2^10 .. 2^20 channels, 4 .. 4096 spectra (odd counts
    among them), 1 .. 16 taps with 8 the most common, either polarisation count, 1 .. 8 sub-bands."""
    lg = rng.randint(10, 20)
    npol = 1 if rng.random() < 0.2 else 2
    nsub, entry = 1, "execute"
    r = rng.random()
    if npol == 2 and r < 0.15 and lg <= 16:
        nsub = rng.choice([2, 4, 8])
    elif r > 0.92:
        entry = "host"
    if rng.random() < 0.65:
        mode = "pfb"
        taps = 8 if rng.random() < 0.6 else rng.choice([2, 4, 6, 12, 16, rng.randint(1, 16)])
        window = rng.choice(["hann", "hann", "hamming", "rect"])
    else:
        mode, taps, window = "direct", 1, rng.choice(["rect", "rect", "hann"])
    nchan = 1 << lg
    room = (1 << 27 if lg <= 18 and taps <= 8 and npol == 2 else 1 << 26) // (nchan * nsub)
    top = max(5, min(4096, room))
    nspectra = min(top, int(round(math.exp(rng.uniform(math.log(4), math.log(top + 1))))))
    return _case(None, nchan, nspectra, mode, taps, npol, window, nsub, entry, rng.choice(["tones", "noise"]))


# ------------------------------------------------------------------ inputs --

def _voltages(n, nchan, npol, nsub, signal, seed):
    """int8 [n][nsub * npol * 2] on the GPU: Gaussian voltages, with polarisations
    correlated and tones in the band, or a weak line over a low noise floor."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    out = torch.empty((n, nsub, npol, 2), dtype=torch.int8, device=DEV)
    sigma = 4.0 if signal == "line" else 20.0
    rho = 0.3 if signal == "tones" else 0.0
    tones = {"noise": [], "line": [(workloads.C4_TONE_AMP, 0.2 * nchan, (0, 1))],
             "tones": [(30.0, 0.1 * nchan + 0.25, (0, 1)), (20.0, 0.37 * nchan + 0.5, (0,))]}[signal]
    tones = [(a, round(b * 4) / 4 if signal == "tones" else float(round(b)), p) for a, b, p in tones]
    block = max(1, (1 << 24) // nsub)
    for m0 in range(0, n, block):
        b = min(block, n - m0)
        v = torch.randn((b, nsub, npol, 2), generator=g, device=DEV) * sigma
        if npol == 2 and rho:
            v[:, :, 1] = rho * v[:, :, 0] + math.sqrt(1.0 - rho * rho) * v[:, :, 1]
        for amp, tbin, pols in tones:
            m = torch.arange(m0, m0 + b, device=DEV, dtype=torch.float64)
            ph = (torch.frac(m * (tbin / nchan)) * (2.0 * math.pi)).float()
            tone = torch.stack([amp * torch.cos(ph), amp * torch.sin(ph)], dim=1)[:, None, :]
            for p in pols:
                if p < npol:
                    v[:, :, p] += tone
        out[m0:m0 + b] = v.round_().clamp_(-127, 127).to(torch.int8)
    return out.view(-1)


def _mode(case):
    return vspec.PFB if case["mode"] == "pfb" else vspec.DIRECT


def _window(case):
    return {"rect": vspec.WIN_RECT, "hann": vspec.WIN_HANN, "hamming": vspec.WIN_HAMMING}[case["window"]]


def _beams():
    """Each beam of the batch as a case of its own."""
    return [_case(None, n, s) if i % 2 == 0 else _case(None, n, s, mode="direct", taps=1, window="rect")
            for i, (n, s) in enumerate(BEAMS)]


def _samples(case):
    return (case["nspectra"] + (case["taps"] if case["mode"] == "pfb" else 1) - 1) * case["nchan"]


def _input(case, seed):
    return _voltages(_samples(case), case["nchan"], case["npol"], case["nsub"], case["signal"], seed)


def prepare(case, seed):
    if case["entry"] == "batch":
        beams = [dict(b, signal=case["signal"]) for b in _beams()]
        batch = vspec.Batch([(b["nchan"], b["taps"], b["npol"], _mode(b), _window(b)) for b in beams])
        ins = [_input(b, seed * 64 + i) for i, b in enumerate(beams)]
        sizes = [batch.out_floats(i) for i in range(len(beams))]
        acc = torch.zeros(sum(sizes), dtype=torch.float32, device=DEV)
        return {"entry": "batch", "batch": batch, "ins": ins, "n": [b["nspectra"] for b in beams], "all": acc,
                "accs": list(acc.split(sizes))}
    plan = vspec.Plan(case["nchan"], case["taps"], case["npol"], _mode(case), _window(case), nsub=case["nsub"])
    x = _input(case, seed)
    if case["entry"] == "host":
        h_in = torch.empty(x.shape, dtype=torch.int8, pin_memory=True)
        h_in.copy_(x)
        h_out = torch.empty(plan.out_floats, dtype=torch.float32, pin_memory=True)
        return {"entry": "host", "plan": plan, "in": h_in, "n": case["nspectra"], "out": h_out}
    acc = torch.zeros(plan.out_floats, dtype=torch.float32, device=DEV)
    return {"entry": "execute", "plan": plan, "in": x, "n": case["nspectra"], "acc": acc}


def run(state):
    if state["entry"] == "batch":
        state["all"].zero_()
        state["batch"].execute(state["ins"], state["n"], state["accs"])
        return state["accs"]
    if state["entry"] == "host":
        state["plan"].execute_host(state["in"], state["n"], state["out"])
        return state["out"]
    state["plan"].dump(state["acc"])  # a new integration: clear the accumulator
    state["plan"].execute(state["in"], state["n"], state["acc"])
    return state["acc"]


def _work(case):
    P = case["taps"] if case["mode"] == "pfb" else 1
    streams = case["npol"] * case["nsub"]
    out = case["nchan"] * case["nsub"] * (16 if case["npol"] == 2 else 4)
    per_sample = (4 * P if case["mode"] == "pfb" else 0) + 5 * math.log2(case["nchan"]) + 8
    return (_samples(case) * streams * 2 + out, per_sample * case["nchan"] * case["nspectra"] * streams)


def work(case):
    parts = [_work(c) for c in (_beams() if case["entry"] == "batch" else [case])]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


# ------------------------------------------------------------ 64-bit values --

def _coefficients(case):
    """h[t][n] in 64 bits: windowed sinc over taps * nchan (PFB) or the window over nchan."""
    N, pfb = case["nchan"], case["mode"] == "pfb"
    L = N * case["taps"] if pfb else N
    i = torch.arange(L, device=DEV, dtype=torch.float64)
    w = torch.ones(L, device=DEV, dtype=torch.float64)
    if case["window"] != "rect":
        a = 0.5 if case["window"] == "hann" else 0.54
        w = a - (1.0 - a) * torch.cos(2.0 * math.pi * i / (L - 1))
    if pfb:
        w = w * torch.sinc((i - 0.5 * (L - 1)) / N)
    return w.view(-1, N)


def _channelize(case, seed):
    N, S, npol, nsub = case["nchan"], case["nspectra"], case["npol"], case["nsub"]
    h = _coefficients(case)
    P = h.shape[0]
    x = _input(case, seed).view(-1, N, nsub, npol, 2)
    res = torch.zeros((nsub, N, 4 if npol == 2 else 1), device=DEV, dtype=torch.float64)
    step = max(1, (1 << 25) // (N * npol))
    for b in range(nsub):
        for s0 in range(0, S, step):
            c = min(step, S - s0)
            spec = []
            for p in range(npol):
                y = torch.zeros((c, N), device=DEV, dtype=torch.complex128)
                for t in range(P):
                    f = x[s0 + t:s0 + t + c, :, b, p, :].to(torch.float64)
                    y += torch.view_as_complex(f.contiguous()) * h[t]
                spec.append(torch.fft.fft(y, dim=1))
            if npol == 1:
                res[b, :, 0] += (spec[0].real ** 2 + spec[0].imag ** 2).sum(0)
            else:
                X, Y = spec
                res[b, :, 0] += (X.real ** 2 + X.imag ** 2).sum(0)
                res[b, :, 1] += (Y.real ** 2 + Y.imag ** 2).sum(0)
                xy = (X * Y.conj()).sum(0)
                res[b, :, 2] += xy.real
                res[b, :, 3] += xy.imag
    return res.view(-1)


def exact(case, seed):
    if case["entry"] == "batch":
        return [_channelize(dict(b, signal=case["signal"]), seed * 64 + i) for i, b in enumerate(_beams())]
    out = _channelize(case, seed)
    return out.cpu() if case["entry"] == "host" else out
