"""The calls a receiver makes of this channelizer, for timing and comparing.

A pass is one call of the public Python binding on data the caller holds: a
chunk of every stream through a plan, many uneven plans in one batch call, the
narrow-band front end with a plan behind it, or chunks in host memory through
the streaming service. Plans, filters and weights are made once, as a receiver
does; a first chunk has gone through them, so the timed chunks have a filled
history. Every pass is the stream's next chunk (its timestamp moves on; the
sample bytes repeat). Shapes are those of workloads.py, the benchmark and the
tests.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2303_09886_gb300 import fengine

PRECISION = {"fp32": fengine.FP32, "fp16": fengine.TC_FP16, "bf16": fengine.TC_BF16}
MAX_DELAY = 4096          # room for coarse delays of 0..2000 samples and their drift over a long run


def _call(name, precision, antennas, channels, taps, spectra, heap=256, rate=1e-9, updates=False, gains=True,
          flags=False, prequant=False):
    return {"name": name, "kind": "call", "precision": precision, "antennas": antennas, "channels": channels,
            "taps": taps, "spectra": spectra, "heap": min(heap, spectra), "rate": rate, "updates": updates,
            "gains": gains, "flags": flags, "prequant": prequant}


def listed():
    return [
        # the smallest call a live receiver makes: 16 spectra of one antenna, latency above all
        _call("lowlat-1k-16sp", "fp32", 1, 1024, 16, 16),
        # the 1024-channel reference configuration, one chunk of 2^20 samples per polarisation
        _call("1k-1ant-2p20", "fp32", 1, 1024, 16, 512, rate=0.0, gains=False),
        # the headline workload: four antennas, 8192 channels, chunks of 2^25 samples
        _call("8k-4ant-2p25-fp32", "fp32", 4, 8192, 16, 2048),
        # the same stream in the FP16 tensor-core form
        _call("8k-4ant-2p25-fp16", "fp16", 4, 8192, 16, 2048),
        # high-bandwidth stream: one antenna, 32768 channels, chunks of 2^28 samples, BF16 form
        _call("32k-1ant-2p28-bf16", "bf16", 1, 32768, 16, 4096, rate=5e-9),
        # the paper's single engine: 32768 channels, chunks of 2^26 samples
        _call("32k-1ant-2p26-fp32", "fp32", 1, 32768, 16, 1024),
        # a ragged chunk of a three-antenna engine with fewer taps: received-heap flags in and out, a last
        # heap that is not full, and fast delays whose model is renewed with every chunk
        _call("4k-3ant-ragged-lost", "fp32", 3, 4096, 8, 1002, heap=100, flags=True, rate=2e-7, updates=True),
        # commissioning: spectra before quantisation are read back to choose the bandpass gains
        _call("2k-2ant-prequant", "fp32", 2, 2048, 16, 515, heap=128, prequant=True),
        # the same in the FP16 form, at 1024 channels
        _call("1k-2ant-prequant-fp16", "fp16", 2, 1024, 8, 640, heap=128, prequant=True),
        # uneven engines of one server in one call: channel counts, taps and chunk lengths differ
        {"name": "batch-24-uneven", "kind": "batch", "members": 24, "min_log2": 18, "max_log2": 22, "mix": 5},
        # narrow-band mode beside the wide-band one: 1/8 of the band into 8192 fine channels
        {"name": "narrowband-d8", "kind": "ddc", "antennas": 2, "decimation": 8, "ddc_taps": 16, "channels": 8192,
         "taps": 16, "spectra": 512},
        # eight antennas' chunks from host memory through the streaming service
        {"name": "service-8ant-8k", "kind": "service", "antennas": 8, "channels": 8192, "taps": 16, "spectra": 128},
    ]


def draw(rng):
    kind = rng.choice(["call"] * 7 + ["batch", "ddc", "service"])
    log2u = lambda lo, hi: 2.0 ** rng.uniform(lo, hi)  # noqa: E731
    if kind == "batch":
        lo = rng.randint(16, 19)
        return {"kind": "batch", "members": rng.randint(3, 40), "min_log2": lo, "max_log2": lo + rng.randint(1, 4),
                "mix": rng.randint(0, 1 << 20)}
    if kind == "ddc":
        d, n = rng.choice([2, 4, 8, 16, 32]), rng.choice([1024, 2048, 4096, 8192])
        ants = rng.randint(1, 3)
        spectra = max(4, int(log2u(18, 24.5) * 2 / (d * ants * 2 * n)))
        return {"kind": "ddc", "antennas": ants, "decimation": d, "ddc_taps": rng.choice([8, 12, 16, 24]),
                "channels": n, "taps": rng.choice([4, 8, 16]), "spectra": spectra}
    if kind == "service":
        n = rng.choice([1024, 4096, 8192])
        return {"kind": "service", "antennas": rng.randint(2, 12), "channels": n, "taps": rng.choice([8, 16]),
                "spectra": max(8, int(log2u(17, 21) / (2 * n)))}
    prec = rng.choice(["fp32"] * 5 + ["fp16", "fp16", "bf16"])
    n, taps = 2 ** rng.randint(8, 15), rng.choice([4, 8, 16, 16, 32])
    if prec != "fp32" and n >= 16384:
        taps = min(taps, 16)
    ants = rng.randint(1, 6)
    # samples of one call over all streams, 2^16 .. 2^28 (2^25 with float spectra out, 2^26 in BF16)
    prequant = rng.random() < 0.2
    total = log2u(16, 25 if prequant else 26 if prec == "bf16" else 28)
    spectra = max(1, int(total / (ants * 4 * n)))
    heap = rng.choice([16, 100, 128, 256])
    rate = rng.choice([0.0, 1e-9, 5e-9, 2e-7] if spectra >= taps else [0.0, 1e-9, 5e-9])   # models are renewed per chunk
    flags = (2 * n * spectra) % fengine.HEAP_SAMPLES == 0 and rng.random() < 0.4
    return {"kind": "call", "precision": prec, "antennas": ants, "channels": n, "taps": taps, "spectra": spectra,
            "heap": min(heap, spectra), "rate": rate, "updates": rate == 2e-7, "gains": rng.random() < 0.8,
            "flags": flags, "prequant": prequant}


# ---- inputs ----

def _rng(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(0x5EED + seed)
    return g


def _samples(g, n, amplitude=60.0):
    """int32 [n] on the GPU: Gaussian noise plus three tones, rounded and clipped to 10 bits."""
    u = torch.rand(10, generator=g, device="cuda", dtype=torch.float64).tolist()
    x = torch.randn(n, generator=g, device="cuda") * (24.0 + 16.0 * u[9])
    i = torch.arange(n, device="cuda", dtype=torch.float64)
    for k in range(3):
        f, a, ph = 0.01 + 0.48 * u[3 * k], 20.0 + amplitude * u[3 * k + 1], u[3 * k + 2]
        x += a * torch.cos(((i * f + ph) % 1.0).float() * (2.0 * math.pi))
    return x.round_().clamp_(-512, 511).to(torch.int32)


def _pack(s):
    """uint8 [5 n / 4]: four samples in five bytes, most significant bit first."""
    u = (s & 0x3FF).view(-1, 4)
    out = torch.empty((u.shape[0], 5), dtype=torch.uint8, device=s.device)
    out[:, 0] = (u[:, 0] >> 2).to(torch.uint8)
    out[:, 1] = (((u[:, 0] & 0x3) << 6) | (u[:, 1] >> 4)).to(torch.uint8)
    out[:, 2] = (((u[:, 1] & 0xF) << 4) | (u[:, 2] >> 6)).to(torch.uint8)
    out[:, 3] = (((u[:, 2] & 0x3F) << 2) | (u[:, 3] >> 8)).to(torch.uint8)
    out[:, 4] = (u[:, 3] & 0xFF).to(torch.uint8)
    return out.view(-1)


def _chunk(g, antennas, samples):
    """uint8 [antenna, pol, 5 L / 4] on the GPU."""
    out = torch.empty((antennas, 2, samples * 5 // 4), dtype=torch.uint8, device="cuda")
    for a in range(antennas):
        for p in range(2):
            out[a, p] = _pack(_samples(g, samples))
    return out


def _models(case, seed):
    """Per antenna the delay and phase, per stream the bandpass gains (complex64)."""
    g = np.random.default_rng([20230317, seed])
    delays = [(float(g.uniform(0, 2000)), float(g.uniform(0, 2 * np.pi))) for _ in range(case["antennas"])]
    n = case["channels"]
    gains = None
    if case.get("gains", True):
        gains = (g.uniform(0.5, 2.0, (case["antennas"], 2, n)) *
                 np.exp(2j * np.pi * g.random((case["antennas"], 2, n)))).astype(np.complex64)
    return delays, gains


def _plan(case, seed, chunk_samples=None):
    n = case["channels"]
    plan = fengine.Plan(case["antennas"], n, case["taps"], chunk_samples or 2 * n * case["spectra"],
                        spectra_per_heap=case.get("heap", 0), max_delay_samples=MAX_DELAY,
                        precision=PRECISION[case.get("precision", "fp32")])
    delays, gains = _models(case, seed)
    for a, (d, ph) in enumerate(delays):
        for p in range(2):
            plan.set_delay(a, p, d, rate=case.get("rate", 1e-9), phase=ph)
            if gains is not None:
                plan.set_gains(a, p, gains[a, p])
    return plan


def _members(case):
    """(channels, taps, chunk samples) of a batch's plans, fixed by the case."""
    g = np.random.default_rng([7, case["mix"]])
    out = []
    for _ in range(case["members"]):
        n, taps = int(g.choice([1024, 4096, 8192, 32768])), int(g.choice([4, 8, 16]))
        length = 2.0 ** g.uniform(case["min_log2"], case["max_log2"])
        out.append((n, taps, 2 * n * max(1, int(length) // (2 * n))))
    return out


class _State:
    pass


def prepare(case, seed):
    s, g, kind = _State(), _rng(seed), case["kind"]
    s.kind, s.t = kind, 0
    if kind == "call":
        s.plan = _plan(case, seed)
        s.rate, s.delays = case["rate"], _models(case, seed)[0] if case["updates"] else []
        s.packed = _chunk(g, case["antennas"], s.plan.chunk_samples)
        s.out = torch.empty(s.plan.info.out_bytes, dtype=torch.int8, device="cuda")
        s.pre = s.valid = s.heap_flags = None
        if case["prequant"]:
            s.pre = torch.empty((case["antennas"], 2, s.plan.M, case["channels"], 2), device="cuda")
        if case["flags"]:
            shape = (case["antennas"], 2, s.plan.chunk_samples // fengine.HEAP_SAMPLES)
            s.valid = (torch.rand(shape, generator=g, device="cuda") > 0.002).to(torch.uint8)
            s.heap_flags = torch.empty((case["antennas"], s.plan.heaps), dtype=torch.uint8, device="cuda")
    elif kind == "batch":
        s.batch, s.plans, s.packed, s.outs = fengine.Batch(8), [], [], []
        for i, (n, taps, length) in enumerate(_members(case)):
            c = {"antennas": 1, "channels": n, "taps": taps}
            s.plans.append(_plan(c, 1000 * seed + i, length))
            s.packed.append(_chunk(g, 1, length))
            s.outs.append(torch.empty(s.plans[-1].info.out_bytes, dtype=torch.int8, device="cuda"))
        s.first = [0] * len(s.plans)
    elif kind == "ddc":
        n, d = case["channels"], case["decimation"]
        length = n * d * case["spectra"]           # 2 n spectra / (2 / D)
        s.ddc = fengine.DDC(case["antennas"], d, case["ddc_taps"], length, 0.2, 1.0)
        s.plan = _plan(case, seed, s.ddc.out_samples)
        s.packed = _chunk(g, case["antennas"], length)
        s.narrow = torch.empty((case["antennas"], 2, s.ddc.out_samples * 5 // 4), dtype=torch.uint8, device="cuda")
        s.out = torch.empty(s.plan.info.out_bytes, dtype=torch.int8, device="cuda")
    else:
        s.service = fengine.Service(8, 8 << 30)
        s.plans, s.h_in, s.h_out = [], [], []
        one = dict(case, antennas=1)
        length = 2 * case["channels"] * case["spectra"]
        for a in range(case["antennas"]):
            s.plans.append(_plan(one, 1000 * seed + a, length))
            s.h_in.append(_chunk(g, 1, length).cpu().pin_memory().numpy())
            s.h_out.append(torch.zeros(s.plans[-1].info.out_bytes, dtype=torch.int8).pin_memory().numpy())
    run(s)                                          # the chunk before: fills the history
    torch.cuda.synchronize()
    return s


def run(s):
    if s.kind == "call":
        for a, (d, ph) in enumerate(s.delays):
            for p in range(2):
                s.plan.set_delay(a, p, d, rate=s.rate, phase=ph, t_apply=s.t, t_ref=s.t)
        s.plan.process(s.packed, s.t, s.out, s.pre, valid=s.valid, heap_flags=s.heap_flags)
        s.t += s.plan.chunk_samples
        return {"out": s.out, "pre": s.pre, "heap_flags": s.heap_flags}
    if s.kind == "batch":
        s.batch.process(list(zip(s.plans, s.packed, s.first, s.outs)))
        s.first = [t + p.chunk_samples for t, p in zip(s.first, s.plans)]
        return s.outs
    if s.kind == "ddc":
        s.ddc.process(s.packed, s.t, s.narrow)
        s.plan.process(s.narrow, s.t * 2 // s.ddc.decimation, s.out)
        s.t += s.ddc.chunk_samples
        return {"narrow": s.narrow, "out": s.out}
    tickets = [s.service.submit(p, h, s.t, o) for p, h, o in zip(s.plans, s.h_in, s.h_out)]
    for t in tickets:
        s.service.wait(t)
    s.t += s.plans[0].chunk_samples
    return s.h_out


# ---- what a pass cannot do without ----

def _plan_work(streams, channels, taps, length):
    """Packed samples in, 8-bit spectra out; FIR, real FFT (2.5 N log2 N), rotation and gain per channel."""
    n = 2.0 * channels
    per_sample = 2.0 * taps + 2.5 * math.log2(n) + 6.0
    return 2.25 * streams * length, per_sample * streams * length


def work(case):
    if case["kind"] == "batch":
        parts = [_plan_work(2, n, taps, length) for n, taps, length in _members(case)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    streams = 2 * case["antennas"]
    if case["kind"] == "ddc":
        out = 2 * case["channels"] * case["spectra"]
        length = out * case["decimation"] // 2
        b, f = _plan_work(streams, case["channels"], case["taps"], out)
        # the narrow-band stream is itself returned, and read back by the plan
        return {"bytes": b + 1.25 * streams * (length + out),
                "flops": f + 4.0 * case["decimation"] * case["ddc_taps"] * streams * out}
    length = 2 * case["channels"] * case["spectra"]
    b, f = _plan_work(streams, case["channels"], case["taps"], length)
    if case.get("prequant"):
        b += 4.0 * streams * length                # n complex floats per 2 n samples
    return {"bytes": b, "flops": f}


# ---- 64 bits ----

def _prototype(channels, taps):
    """Hann-windowed sinc of 2 n T points, sum of squares 1, as the plan holds it (rounded to 32 bits)."""
    size, n = 2 * channels * taps, 2 * channels
    u = np.arange(size) + 0.5
    w = np.sin(np.pi * u / size) ** 2 * np.sinc((u - size / 2) / n)
    return torch.from_numpy((w / np.sqrt(np.sum(w * w))).astype(np.float32)).cuda().double()


def exact(case, seed):
    """Spectra before quantisation of the pass after prepare(): the chunk at
    t = L of a stream that starts at 0 with the same chunk. The 8-bit and
    packed outputs are whole numbers."""
    if case["kind"] != "call" or not case["prequant"]:
        return None
    n, taps, m = case["channels"], case["taps"], case["spectra"]
    size, length = 2 * n, 2 * n * m
    g = _rng(seed)
    delays, gains = _models(case, seed)
    w = _prototype(n, taps)
    pre = torch.empty((case["antennas"], 2, m, n, 2), dtype=torch.float64, device="cuda")
    lead = size * taps + 2 * MAX_DELAY             # zeros before the stream's first sample
    t0 = size * torch.arange(length // size - taps + 1, length // size - taps + 1 + m, device="cuda",
                             dtype=torch.int64)
    k = torch.arange(n, device="cuda", dtype=torch.float64)
    at = torch.arange(size, device="cuda")
    for a, (delay, phase) in enumerate(delays):
        t_ref = torch.where(t0 >= length, length, 0) if case["updates"] else 0
        d = delay + case["rate"] * (t0 - t_ref).double()
        c = torch.floor(d + 0.5)
        rot = phase - 2 * math.pi * ((d - c)[:, None] * k / size)
        for p in range(2):
            x = _samples(g, length).double()
            x = torch.cat([torch.zeros(lead, dtype=torch.float64, device="cuda"), x, x])
            y = torch.zeros((m, size), dtype=torch.float64, device="cuda")
            start = (t0 - c.long() + lead)[:, None] + at
            for j in range(taps):
                y += w[size * j:size * (j + 1)] * x[start + size * j]
            f = torch.fft.rfft(y, dim=1)[:, :n] * torch.polar(torch.ones_like(rot), rot)
            if gains is not None:
                f = f * torch.from_numpy(gains[a, p].astype(np.complex128)).cuda()
            pre[a, p] = torch.view_as_real(f)
    return {"out": None, "pre": pre, "heap_flags": None}
