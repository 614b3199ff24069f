"""The calls whose speed matters to a user of the fan-beam library.

Each case is a call (or the few calls that belong together) as a program makes
them through ``paper_1702_04728_gb300.binding``: baseband requests of one coarse
channel up to the whole band, through each precision form, as one request, as a
stream cut anywhere, with tracking E-W beams and as a mix of many streams on a
serving plan; and the products made of the intensity output.

Voltages are noise of 2.5 counts per part plus a plane wave, quantised to 4 + 4
bits; intensities are sums of 48 chi-squared terms with a bright pulse.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1702_04728_gb300 import binding as B

FORMS = {"fp32": B.BF_FP32_FFT, "tc3": B.BF_TC_DFT256, "tc2": B.BF_TC_DFT256_X2, "tc1": B.BF_TC_DFT256_X1,
         "tc512": B.BF_TC_DFT512}
FRAME, INPUTS, BEAMS = B.FRAME, B.N_INPUT, B.N_BEAMS
MOST = 1024 * 768            # channel-samples of the largest request: the 1024-channel band for two frames

# What separates two correct implementations of a form, as (relative 2-norm, largest).  The 32-bit
# forms differ by the order of ~20 rounded operations per term and of 96 terms per output (1.2e-7 of
# the result from 64 bits in the FFT form, 3.8e-6 in the 3-term GEMM, whose tensor core truncates its
# 32-bit sums); the 2- and 1-term forms by the FP16 rounding of twiddles, or of twiddles and data
# (up to 6.4e-5; the largest single difference is some ten times that).  Four times what was measured.
BEAM_TOL = {"fp32": (5e-7, 4e-6), "tc3": (1.6e-5, 6e-5), "tc2": (2.5e-4, 2e-3), "tc1": (2.5e-4, 2e-3),
            "tc512": (2.5e-4, 2e-3)}


def listed():
    return [
        # one frame (0.98 ms) of one channel: the shortest request, as a latency-bound trigger makes it
        {"name": "frame", "kind": "request", "form": "fp32", "n_chan": 1, "n_samples": 384, "track": False},
        # eight frames of one channel with some samples over: a short look at a source
        {"name": "source", "kind": "request", "form": "fp32", "n_chan": 1, "n_samples": 3089, "track": False},
        # a correlator node's share: four channels, 126 ms; the library's headline workload
        {"name": "slice", "kind": "request", "form": "fp32", "n_chan": 4, "n_samples": 49152, "track": False},
        # all 1024 channels for two frames: wide and short, many launches' worth of channels
        {"name": "band", "kind": "request", "form": "fp32", "n_chan": 1024, "n_samples": 768, "track": False},
        # a live stream: ragged packets whose leftover samples carry over, beams that follow the sky
        {"name": "stream", "kind": "stream", "form": "fp32", "n_chan": 3, "n_samples": 20011, "pieces": 5,
         "track": True},
        # many users' streams of uneven length on one serving plan
        {"name": "serving", "kind": "serving", "form": "fp32", "streams": 24, "max_chan": 8, "max_frames": 20,
         "mix": 1},
        # the node's share through the tensor-core forms: 32-bit class error ...
        {"name": "slice_tc3", "kind": "request", "form": "tc3", "n_chan": 4, "n_samples": 49152, "track": False},
        # ... one channel at FP16 twiddles ...
        {"name": "channel_tc2", "kind": "request", "form": "tc2", "n_chan": 1, "n_samples": 49152, "track": False},
        # ... the fastest form ...
        {"name": "slice_tc1", "kind": "request", "form": "tc1", "n_chan": 4, "n_samples": 49152, "track": False},
        # ... and one channel through the full zero-padded transform
        {"name": "channel_tc512", "kind": "request", "form": "tc512", "n_chan": 1, "n_samples": 49152,
         "track": False},
        # the 8-bit archive product of a node's output
        {"name": "codes", "kind": "codes", "n_sub": 64, "n_frames": 128},
        # search products of one second of 64 channels: one dedispersed series per beam, and the sky map
        {"name": "search", "kind": "search", "n_chan": 64, "n_frames": 1017, "dm": 20.0},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    kind = rng.choice(["request", "request", "request", "stream", "serving", "codes", "search"])
    if kind in ("request", "stream"):
        n_chan = _log_int(rng, 1, 1024 if kind == "request" else 16)
        n = _log_int(rng, FRAME, min(60000, MOST // n_chan))
        case = {"kind": kind, "form": rng.choice(["fp32", "fp32"] + list(FORMS)), "n_chan": n_chan, "n_samples": n,
                "track": rng.random() < 0.25}
        if kind == "stream":
            case["pieces"] = rng.randint(2, 8)
        return case
    if kind == "serving":
        return {"kind": kind, "form": rng.choice(["fp32", "fp32"] + list(FORMS)), "streams": rng.randint(4, 24),
                "max_chan": rng.randint(1, 8), "max_frames": rng.randint(1, 20), "mix": rng.randrange(1 << 20)}
    if kind == "codes":
        n_sub = 16 * _log_int(rng, 1, 1024)
        return {"kind": kind, "n_sub": n_sub, "n_frames": _log_int(rng, 2, min(2048, (1 << 26) // (BEAMS * n_sub) + 2))}
    n_chan = _log_int(rng, 2, 64)
    return {"kind": kind, "n_chan": n_chan, "n_frames": _log_int(rng, 64, 1024), "dm": round(rng.uniform(0.0, 1.2), 3)}


# ---- inputs ---------------------------------------------------------------------------------

def _freqs(n_chan):
    return [400e6 + 400e6 * (i + 0.5) / n_chan for i in range(n_chan)]


def _voltages(n_chan, n_samples, gen, freqs):
    """uint8 [n_chan][n_samples][2048] on the GPU: noise and a plane wave with a random phase per sample."""
    out = torch.empty((n_chan, n_samples, INPUTS), dtype=torch.uint8, device="cuda")
    u, s = torch.rand(2, generator=gen, device="cuda").tolist()
    u, s = 0.02 * (u - 0.5), 1.6 * (s - 0.5)
    path = (torch.arange(4, device="cuda", dtype=torch.float64).view(4, 1) * (20.0 * u)
            + torch.arange(256, device="cuda", dtype=torch.float64) * (0.3048 * s)).view(-1)
    step = max(1, (1 << 26) // INPUTS)
    for c, f in enumerate(freqs):
        ph = (2 * math.pi * torch.remainder(path * (f / 299792458.0), 1.0)).float().view(1, -1, 1)
        for t0 in range(0, n_samples, step):
            n = min(step, n_samples - t0)
            turn = 2 * math.pi * torch.rand((n, 1, 2), generator=gen, device="cuda")
            parts = []
            for wave in (torch.cos(ph + turn), torch.sin(ph + turn)):
                v = torch.randn((n, 1024, 2), generator=gen, device="cuda").mul_(2.5).add_(wave)
                parts.append(v.round_().clamp_(-7, 7).add_(8).to(torch.uint8))
            out[c, t0:t0 + n] = (parts[0] * 16 + parts[1]).view(n, INPUTS)
    return out


def _intensities(n_sub, n_frames, gen):
    x = torch.randn((BEAMS, n_sub, n_frames), generator=gen, device="cuda")
    x.mul_(math.sqrt(48.0)).add_(48.0).clamp_(min=1.0).mul_(1e4)
    x[::7, :, n_frames // 3] *= 3.0
    return x


def _sines(n_frames, rng):
    """E-W sines of four beams that drift with the sky, one row per output frame."""
    t = np.arange(n_frames, dtype=np.float64)[:, None]
    return np.sin(np.radians(np.array([-0.6, -0.2, 0.2, 0.6]) + rng.uniform(-0.3, 0.3) + 4e-6 * t))


def _lengths(case):
    """The stream's packets: n_samples cut at random places."""
    rng = random.Random(case["n_samples"] * 16 + case["pieces"])
    cuts = sorted(rng.randint(0, case["n_samples"]) for _ in range(case["pieces"] - 1))
    return [b - a for a, b in zip([0] + cuts, cuts + [case["n_samples"]])]


def _mix(case):
    """(channels, samples) of every request of the serving mix."""
    rng = random.Random(case["mix"])
    return [(rng.randint(1, case["max_chan"]), FRAME * rng.randint(1, case["max_frames"]) + rng.randint(0, FRAME - 1))
            for _ in range(case["streams"])]


def _mix_freqs(n_chan, i):
    return [400e6 + 390625.0 * ((37 * i + 101 * c) % 1024 + 0.5) for c in range(n_chan)]


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    rng = random.Random(seed)
    kind = case["kind"]
    if kind in ("request", "stream"):
        freqs = _freqs(case["n_chan"])
        vin = _voltages(case["n_chan"], case["n_samples"], gen, freqs)
        return freqs, vin, _sines(case["n_samples"] // FRAME, rng) if case["track"] else None
    if kind == "serving":
        out = []
        for i, (c, n) in enumerate(_mix(case)):
            freqs = _mix_freqs(c, i)
            out.append((freqs, _voltages(c, n, gen, freqs)))
        return out
    return _intensities(case["n_sub"] if kind == "codes" else 16 * case["n_chan"], case["n_frames"], gen)


# ---- what a program has in hand, and the call ---------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind}
    data = _inputs(case, seed)
    if kind in ("request", "stream"):
        st["freqs"], vin, st["track"] = data
        st["plan"] = B.Plan(form=FORMS[case["form"]])
        if kind == "request":
            st["vin"] = vin
        else:
            st["packets"], a, carry = [], 0, 0
            for n in _lengths(case):
                nf = (carry + n) // FRAME
                out = torch.empty((BEAMS, 16 * case["n_chan"], nf), dtype=torch.float32, device="cuda")
                st["packets"].append((vin[:, a:a + n].contiguous(), n, nf, out))
                carry = (carry + n) % FRAME
                a += n
    elif kind == "serving":
        st["plan"] = B.Plan(mode=B.BF_MODE_SERVING, stream=None, form=FORMS[case["form"]])
        st["requests"] = [(freqs, vin, torch.empty((BEAMS, 16 * len(freqs), vin.shape[1] // FRAME),
                                                   dtype=torch.float32, device="cuda")) for freqs, vin in data]
    else:
        st["plan"] = B.Plan()
        st["x"] = data
        if kind == "search":
            st["freqs"], st["dm"] = _freqs(case["n_chan"]), case["dm"]
    torch.cuda.synchronize()         # a serving plan runs on a stream of its own
    return st


def run(st):
    plan, kind = st["plan"], st["kind"]
    if kind == "request":
        return plan.run(st["vin"], st["freqs"], ew_sin_frames=st["track"])
    if kind == "stream":
        # packets are submitted as they come; the results are collected once the stream has ended
        tickets, first = [], 0
        for i, (vin, n, nf, out) in enumerate(st["packets"]):
            rows = None if st["track"] is None else st["track"][first:first + nf]
            last = i + 1 == len(st["packets"])
            tickets.append(plan.submit(vin, st["freqs"], out if nf else None, stream_id=1,
                                       flags=B.BF_END_OF_STREAM if last else 0, n_samples=n,
                                       ew_sin_frames=rows if nf else None)[1])
            first += nf
        for t in tickets:
            plan.poll(t)
        return [p[3] for p in st["packets"] if p[2]]
    if kind == "serving":
        tickets = [plan.submit(vin, freqs, out, stream_id=100 + i, flags=B.BF_END_OF_STREAM)[1]
                   for i, (freqs, vin, out) in enumerate(st["requests"])]
        for t in tickets:
            plan.poll(t)
        return [out for _, _, out in st["requests"]]
    if kind == "codes":
        return plan.rescale_u8(st["x"])
    return plan.dedisperse(st["x"], st["freqs"], st["dm"]), plan.skymap(st["x"])


# ---- what a pass cannot do without ------------------------------------------------------------

def _shapes(case):
    """(channels, samples) of the case's baseband requests."""
    if case["kind"] == "serving":
        return _mix(case)
    return [(case["n_chan"], case["n_samples"])]


def work(case):
    kind = case["kind"]
    if kind in ("request", "stream", "serving"):
        nbytes = flops = 0
        for c, n in _shapes(case):
            nf = n // FRAME
            nbytes += c * (nf * FRAME * INPUTS + 4 * BEAMS * 16 * nf)
            # per input-sample: N-S 512-point FFT 90, E-W beams 32, 128-point FFT 35, detection 5
            flops += 162 * c * nf * FRAME * INPUTS
        return {"bytes": nbytes, "flops": flops}
    if kind == "codes":
        n = BEAMS * case["n_sub"] * case["n_frames"]
        return {"bytes": 5 * n + 8 * BEAMS * case["n_sub"], "flops": 7 * n}
    n = BEAMS * 16 * case["n_chan"] * case["n_frames"]
    n_out = max(0, case["n_frames"] - int(_delays(case).max()))
    return {"bytes": 4 * (n + BEAMS * (n_out + 1)), "flops": n + BEAMS * 16 * case["n_chan"] * n_out}


def tolerance(case):
    kind = case["kind"]
    if kind in ("request", "stream", "serving"):
        rel, big = BEAM_TOL[case["form"]]
        return {"rel": rel, "max": big}
    if kind == "codes":
        # 32-bit means and deviations; a code next to a rounding boundary may fall on either side
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.002}
    return {"rel": 4e-6, "max": 2e-5}         # 32-bit sums: 4.4e-7 from 64 bits over 1024 sub-channels


# ---- 64-bit results -----------------------------------------------------------------------------

def _exact_channel(raw, f, sines):
    """[1024][16][n_frames] of one channel: direct definition in 64 bits (raw: uint8 [n][2048])."""
    nf = raw.shape[0] // FRAME
    m = (np.arange(256) - 127.5) / 128.0
    lut = np.floor((((512.0 * f) * 0.3048) * m) / 299792458.0 + 0.5).astype(np.int64) % 512
    lut = torch.from_numpy(lut).cuda()
    if sines is None:
        sines = np.broadcast_to(np.sin(np.array([-0.6, -0.2, 0.2, 0.6]) * math.pi / 180.0), (nf, 4))
    turns = (f * np.arange(4.0) * 20.0) * sines[:, :, None] / 299792458.0          # [frame][beam][cylinder]
    w = torch.from_numpy(np.exp(-2j * math.pi * (turns - np.floor(turns)))).cuda()
    out = torch.empty((BEAMS, 16, nf), dtype=torch.float64, device="cuda")
    for a in range(0, nf, 16):
        k = min(16, nf - a)
        b = raw[a * FRAME:(a + k) * FRAME]
        x = torch.complex((b >> 4).double() - 8, (b & 15).double() - 8).view(k, FRAME, 4, 256, 2)
        y = torch.einsum("fjc,ftcnp->fjptn", w[a:a + k], x)
        y = torch.fft.fft(y, n=512, dim=-1).index_select(-1, lut)                  # [f][j][p][t][m]
        y = torch.fft.fft(y.view(k, 4, 2, 3, 128, 256), dim=4)
        z = (y.real ** 2 + y.imag ** 2).sum(dim=(2, 3))                            # [f][j][q][m]
        z = torch.fft.fftshift(z, dim=2).view(k, 4, 16, 8, 256).sum(dim=3)
        out[:, :, a:a + k] = z.permute(1, 3, 2, 0).reshape(BEAMS, 16, k)
    return out


def _exact_request(freqs, vin, sines):
    return torch.cat([_exact_channel(vin[c], f, sines) for c, f in enumerate(freqs)], dim=1)


def _delays(case):
    fine = 390625.0 / 128
    f = np.array([[(c + (8 * s + 3.5 - 64) * fine) / 1e6 for s in range(16)] for c in _freqs(case["n_chan"])]).ravel()
    x = ((4.148808e3 * case["dm"]) * (1.0 / (f * f) - 1.0 / (f.max() * f.max()))) / (384 * 2.56e-6)
    return np.floor(x + 0.5).astype(np.int64)


def exact(case, seed):
    kind = case["kind"]
    data = _inputs(case, seed)
    if kind == "request":
        return _exact_request(*data)
    if kind == "stream":
        whole, first, carry, outs = _exact_request(*data), 0, 0, []
        for n in _lengths(case):
            nf = (carry + n) // FRAME
            carry = (carry + n) % FRAME
            if nf:
                outs.append(whole[:, :, first:first + nf].contiguous())
            first += nf
        return outs
    if kind == "serving":
        return [_exact_request(freqs, vin, None) for freqs, vin in data]
    if kind == "codes":
        n = data.shape[2]
        stats = torch.empty((BEAMS, data.shape[1], 2), dtype=torch.float64, device="cuda")
        for b in range(0, BEAMS, 64):
            x = data[b:b + 64].double()
            stats[b:b + 64, :, 0] = x.sum(dim=2) / n
            stats[b:b + 64, :, 1] = x.var(dim=2, unbiased=False).sqrt()
        return None, stats
    d = _delays(case)
    n_out = max(0, case["n_frames"] - int(d.max()))
    series = torch.zeros((BEAMS, n_out), dtype=torch.float64, device="cuda")
    for s in range(len(d)):
        series += data[:, s, int(d[s]):int(d[s]) + n_out]
    return series, torch.stack([data[b].double().sum() for b in range(BEAMS)])
