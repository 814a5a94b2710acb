"""The workloads that performance work on this package is measured on.

Each case is one call, or one short run of calls, that a survey pipeline
makes: a transform of one beam (float32, uint8 or float32 with fp16 state), a
differentiable step, a transform with its pulse search, the spectra from
voltages, a batch of uneven beams, or a stream in chunks.  ``listed`` names
the cases; ``draw`` gives further ones of the same ranges (channels, samples,
delays, data types, channel order and delay offset).  Inputs are N(0, 1)
noise with dispersed pulses of 0.5 .. 2 sigma per channel, as uint8 scaled to
128 + 16 x and clipped, made on the device from the seed.

``exact`` computes the same outputs in 64 bits with plain torch, straight
from the definition: Option-1 partial sums per channel, then one addition per
row and merge level (section 4 of arXiv:1411.5373).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1411_5373_gb300 as fdmt

LARGEST_CELLS = 4096 * (1 << 18)  # rows x samples of the largest beam measured


def _beam(name, nf, nt, nd, dtype, f_min=1200.0, f_max=1600.0, **more):
    return {"name": name, "kind": "beam", "nf": nf, "nt": nt, "nd": nd, "dtype": dtype, "f_min": f_min,
            "f_max": f_max, "schedule": "fused", "d_min": 0, "descending": False, **more}


def listed():
    return [
        # The smallest useful beam, as an interactive user or a trigger on a
        # short buffer runs it: latency and launches are what it costs.
        _beam("beam-64-f32", 64, 1024, 64, "f32"),
        # A sub-band of a low-latency search: few channels, a short buffer.
        _beam("beam-256-u8", 256, 16384, 512, "u8"),
        # The standard beam (a 400 MHz band in 1024 channels, 1024 trial
        # delays), float32 filterbanks after cleaning.
        _beam("beam-1k-f32", 1024, 65536, 1024, "f32"),
        # The same straight from an 8-bit filterbank file, exact sums.
        _beam("beam-1k-u8", 1024, 65536, 1024, "u8"),
        # The same with the stored state in fp16, for callers short of memory.
        _beam("beam-1k-f16state", 1024, 65536, 1024, "f16state"),
        # A real file: masked channels cut off (not a power of two), an odd
        # length, highest channel first, delays from 500 samples up.
        _beam("beam-1000-ragged-f32", 1000, 50004, 777, "f32", d_min=500, descending=True),
        # A wide band at full resolution with 4096 delays: the largest beam.
        _beam("beam-4k-f32", 4096, 1 << 18, 4096, "f32", 1100.0, 1700.0),
        # One optimisation step on channel weights and input: transform,
        # adjoint and weight gradient through autograd.
        {**_beam("step-1k-f32", 1024, 65536, 1024, "f32"), "kind": "step"},
        # Detection: the transform, then peak and time per delay for widths
        # 1 .. 128 samples.
        {**_beam("search-1k-f32", 1024, 65536, 1024, "f32"), "kind": "search", "widths": 8},
        # The front end: 64 M complex voltages to 1024 channels.
        {"name": "filterbank-1k", "kind": "filterbank", "nf": 1024, "nt": 65536, "nbin": 1},
        # A multi-beam receiver's beams of different shapes in one call.
        {"name": "batch-8-u8", "kind": "batch", "beams": 8, "beams_seed": 1, "dtype": "u8", "f_min": 1200.0,
         "f_max": 1600.0, "schedule": "launches"},
        # Real-time operation: four chunks of a continuous 8-bit stream.
        {"name": "stream-1k-u8", "kind": "stream", "nf": 1024, "chunk": 16384, "nd": 1024, "pushes": 4,
         "dtype": "u8", "f_min": 1200.0, "f_max": 1600.0, "schedule": "fused"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_beam(rng):
    """A beam of any size in the range whose rows stay below the largest's."""
    dtype = rng.choice(["f32", "f32", "u8", "f16state"])
    quantum = {"f32": 4, "u8": 16, "f16state": 8}[dtype]  # rows are whole 16-byte words
    nf = 2 ** rng.randint(5, 12) if rng.random() < 0.5 else _log_int(rng, 24, 4000)
    nt = 2 ** rng.randint(10, 18) if rng.random() < 0.4 else _log_int(rng, 1000, 200000) // quantum * quantum
    nd = min(nt, _log_int(rng, 32, 4096))
    while max(nf, nd) * nt > LARGEST_CELLS // 2:
        nt = nt // 2 // quantum * quantum
        nd = min(nd, nt)
    band = rng.choice([(1200.0, 1600.0), (1100.0, 1700.0)])
    mapped = rng.random() < 0.25
    return _beam("", nf, nt, nd, dtype, *band, d_min=rng.randint(1, 1000) if mapped else 0,
                 descending=mapped and rng.random() < 0.5)


def draw(rng):
    kind = rng.choice(["beam"] * 6 + ["step", "search", "filterbank", "batch", "stream"])
    if kind == "filterbank":
        nf, nbin = 2 ** rng.randint(5, 12), rng.choice([1, 1, 2, 4])
        case = {"kind": kind, "nf": nf, "nt": _log_int(rng, 100, (1 << 26) // (nf * nbin)), "nbin": nbin}
    elif kind == "batch":
        case = {"kind": kind, "beams": rng.randint(2, 8), "beams_seed": rng.randint(2, 10 ** 6), "dtype": "u8",
                "f_min": 1200.0, "f_max": 1600.0, "schedule": "launches"}
    elif kind == "stream":
        case = {"kind": kind, "nf": 2 ** rng.randint(6, 11), "chunk": _log_int(rng, 1024, 65536) // 16 * 16,
                "nd": _log_int(rng, 64, 2048), "pushes": rng.randint(2, 5), "dtype": rng.choice(["u8", "f32"]),
                "f_min": 1200.0, "f_max": 1600.0, "schedule": "fused"}
    else:
        case = _draw_beam(rng)
        if kind == "step":
            case.update(kind=kind, dtype="f32", nt=min(case["nt"], 1 << 16))
            case["nd"] = min(case["nd"], case["nt"])
        elif kind == "search":
            case.update(kind=kind, widths=rng.randint(1, 10))
    case.pop("name", None)
    return case


def _beams(case):
    """(nf, nt, nd) of the beams of a batch."""
    rng = np.random.default_rng(case["beams_seed"])
    out = []
    for _ in range(case["beams"]):
        nf = int(rng.choice([256, 512, 1024]))
        nt = int(rng.choice([1 << 14, 1 << 16]))
        out.append((nf, nt, int(rng.choice([256, 512, 1024]))))
    return out


# ---- inputs --------------------------------------------------------------

def _signal(nf, nt, nd, f_min, f_max, gen):
    """Noise with eight dispersed pulses, float32 on the device."""
    x = torch.randn((nf, nt), generator=gen, device="cuda")
    edges = torch.linspace(f_min, f_max, nf + 1, dtype=torch.float64, device="cuda")[:-1]
    r = (f_min ** -2 - edges ** -2) / (f_min ** -2 - f_max ** -2)
    host = torch.rand((8, 4), generator=gen, device="cuda").cpu()
    rows = torch.arange(nf, device="cuda")[:, None]
    for u in host.tolist():
        width = 1 + int(u[0] * 16)
        at = (u[1] * nt - (u[2] * nd * r).round()).long()[:, None] + torch.arange(width, device="cuda")
        inside = (at >= 0) & (at < nt)
        x[rows.expand_as(at)[inside], at[inside]] += 0.5 + 1.5 * u[3]
    return x


def _input(nf, nt, nd, f_min, f_max, dtype, gen):
    x = _signal(nf, nt, nd, f_min, f_max, gen)
    return (128.0 + 16.0 * x).round_().clamp_(0, 255).to(torch.uint8) if dtype == "u8" else x


def _inputs(case, seed):
    """What a user holds before the call, without plans: a dict of tensors."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    if kind == "filterbank":
        n = case["nf"] * case["nt"] * case["nbin"]
        return {"volts": torch.view_as_complex(torch.randn((n, 2), generator=gen, device="cuda"))}
    if kind == "batch":
        return {"x": [_input(*b, case["f_min"], case["f_max"], case["dtype"], gen) for b in _beams(case)]}
    if kind == "stream":
        x = _input(case["nf"], case["chunk"] * case["pushes"], case["nd"], case["f_min"], case["f_max"],
                   case["dtype"], gen)
        return {"x": [c.contiguous() for c in x.split(case["chunk"], dim=1)]}
    got = {"x": _input(case["nf"], case["nt"], case["nd"], case["f_min"], case["f_max"], case["dtype"], gen)}
    if kind == "step":
        got["w"] = 0.5 + torch.rand(case["nf"], generator=gen, device="cuda")
        got["g"] = torch.randn((case["nd"], case["nt"]), generator=gen, device="cuda")
    return got


def prepare(case, seed):
    state = {"case": case, **_inputs(case, seed)}
    kind = case["kind"]
    if kind == "batch":
        beams = [(case["f_min"], case["f_max"], *b) for b in _beams(case)]
        state["plan"] = fdmt.BatchPlan(beams, case["dtype"], schedule=case["schedule"])
        state["out"] = state["plan"].outputs()
        state["plan"].workspace()
    elif kind == "stream":
        state["plan"] = fdmt.Stream(case["f_min"], case["f_max"], case["nf"], case["chunk"], case["nd"],
                                    dtype=case["dtype"], schedule=case["schedule"])
    elif kind != "filterbank":
        state["plan"] = fdmt.Plan(case["f_min"], case["f_max"], case["nf"], case["nt"], case["nd"],
                                  dtype=case["dtype"], schedule=case["schedule"], d_min=case["d_min"],
                                  descending=case["descending"])
        state["plan"].workspace()
    if kind == "step":
        state["plan"].adjoint_workspace()
        state["x"].requires_grad_(True)
        state["w"].requires_grad_(True)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "filterbank":
        return fdmt.filterbank(state["volts"], case["nf"], case["nbin"])
    plan, x = state["plan"], state["x"]
    if kind == "batch":
        return plan.execute(x, state["out"])
    if kind == "stream":
        plan.reset()
        return [plan.push(c) for c in x]
    if kind == "step":
        out = fdmt.fdmt(x, plan, state["w"])
        gx, gw = torch.autograd.grad(out, (x, state["w"]), state["g"])
        return {"out": out.detach(), "grad_x": gx, "grad_w": gw}
    out = plan.execute(x)
    if kind == "search":
        peak, time = plan.search(out, case["widths"])
        return {"out": out, "peak": peak, "time": time}
    return out


# ---- what a pass cannot do without ---------------------------------------

def _tables(f_min, f_max, nf, nd):
    """(lower row, upper row or -1, shift) of every row per merge level, and
    the Option-1 rows per channel: the addition rule's integer tables."""
    levels = (nf - 1).bit_length()
    edge = [f_min + (f_max - f_min) * k / nf for k in range(nf + 1)]
    rows, merges = [nd], []
    for level in range(levels, 0, -1):
        child, lows = [], []
        for b, r in enumerate(rows):
            k0, k1, k2 = b << level, (b << level) + (1 << (level - 1)), min((b + 1) << level, nf)
            if k1 >= nf:
                child.append(r)
                lows.append((np.arange(r), None))
                continue
            i0, i1, i2 = (1.0 / (edge[k] * edge[k]) for k in (k0, k1, k2))
            low = np.floor((i0 - i1) / (i0 - i2) * np.arange(r) + 0.5).astype(np.int64)
            child += [int(low[-1]) + 1, r - 1 - int(low[-1]) + 1]
            lows.append((low, np.arange(r) - low))
        start = np.concatenate(([0], np.cumsum(child)))
        lo, hi, shift, c = [], [], [], 0
        for low, high in lows:
            lo.append(start[c] + low)
            hi.append(np.full(len(low), -1) if high is None else start[c + 1] + high)
            shift.append(low)
            c += 1 if high is None else 2
        merges.insert(0, tuple(np.concatenate(v) for v in (lo, hi, shift)))
        rows = child
    return rows, merges


def _adds(case_or_shape, nf, nt, nd):
    rows, merges = _tables(*case_or_shape, nf, nd)
    return float(nt) * (sum(rows) + sum(len(m[0]) for m in merges))


def work(case):
    kind = case["kind"]
    if kind == "filterbank":
        n = float(case["nf"]) * case["nt"] * case["nbin"]
        return {"bytes": 8 * n + 4.0 * case["nf"] * case["nt"], "flops": n * (5 * math.log2(case["nf"]) + 3)}
    es = 1 if case["dtype"] == "u8" else 4
    band = (case["f_min"], case["f_max"])
    if kind == "batch":
        return {"bytes": float(sum(nf * nt * es + nd * nt * 4 for nf, nt, nd in _beams(case))),
                "flops": sum(_adds(band, *b) for b in _beams(case))}
    nf, nd = case["nf"], case["nd"]
    nt = case["chunk"] * case["pushes"] if kind == "stream" else case["nt"]
    size, adds = float(nf * nt * es + nd * nt * 4), _adds(band, nf, nt, nd)
    if kind == "step":  # also the gradient in, the input's gradient out, the input for the weights' gradient
        return {"bytes": size + 4.0 * nt * (nd + 2 * nf), "flops": 2 * adds + 3.0 * nf * nt}
    if kind == "search":  # also one sum and one comparison per value and width
        return {"bytes": size, "flops": adds + 2.0 * nd * nt * case["widths"]}
    return {"bytes": size, "flops": adds}


# ---- the outputs in 64 bits ------------------------------------------------

def _transform64(x, band, nd):
    rows, merges = _tables(*band, x.shape[0], nd)
    nt = x.shape[1]
    state = x.double().repeat_interleave(torch.tensor(rows, device=x.device), dim=0)
    at = 0
    for r in rows:  # row j adds the channel's samples one .. j earlier
        for j in range(1, r):
            state[at + j] = state[at + j - 1]
            state[at + j, j:] += state[at, :nt - j]
        at += r
    for lo, hi, shift in merges:
        new = state[torch.from_numpy(lo).to(x.device)]
        for row, (h, s) in enumerate(zip(hi.tolist(), shift.tolist())):
            if h >= 0 and s < nt:
                new[row, s:] += state[h, :nt - s]
        state = new
    return state


def _adjoint64(g, band, nf):
    rows, merges = _tables(*band, nf, g.shape[0])
    nt = g.shape[1]
    grad = g.double()
    for level in range(len(merges) - 1, -1, -1):
        lo, hi, shift = merges[level]
        below = len(merges[level - 1][0]) if level else sum(rows)
        new = torch.zeros((below, nt), dtype=torch.float64, device=g.device)
        for row, (l, h, s) in enumerate(zip(lo.tolist(), hi.tolist(), shift.tolist())):
            new[l] += grad[row]
            if h >= 0 and s < nt:
                new[h, :nt - s] += grad[row, s:]
        grad = new
    out = torch.zeros((nf, nt), dtype=torch.float64, device=g.device)
    at = 0
    for k, r in enumerate(rows):
        for i in range(min(r, nt)):  # every row j >= i takes the sample i earlier
            out[k, :nt - i] += grad[at + i:at + r, i:].sum(dim=0)
        at += r
    return out


def _mapped(x, case):
    """The input in channel order, each channel delayed by its share of d_min."""
    nf, nt = x.shape
    f0, f1 = case["f_min"], case["f_max"]
    x = x.flip(0) if case["descending"] else x
    if case["d_min"] == 0:
        return x
    out = torch.zeros_like(x)
    for k in range(nf):
        f = f0 + (f1 - f0) * k / nf
        s = math.floor(case["d_min"] * ((f0 ** -2 - f ** -2) / (f0 ** -2 - f1 ** -2)) + 0.5)
        if s < nt:
            out[k, s:] = x[k, :nt - s]
    return out


def _unmapped(g, case):
    """The transpose of _mapped."""
    nf, nt = g.shape
    f0, f1 = case["f_min"], case["f_max"]
    out = torch.zeros_like(g)
    for k in range(nf):
        f = f0 + (f1 - f0) * k / nf
        s = math.floor(case["d_min"] * ((f0 ** -2 - f ** -2) / (f0 ** -2 - f1 ** -2)) + 0.5)
        if s < nt:
            out[k, :nt - s] = g[k, s:]
    return out.flip(0) if case["descending"] else out


def _like(out64, dtype):
    return out64.round().to(torch.int32) if dtype == "u8" else out64


def exact(case, seed):
    got = _inputs(case, seed)
    kind = case["kind"]
    if kind == "filterbank":
        nf, nt, nbin = case["nf"], case["nt"], case["nbin"]
        power = torch.zeros((nt, nf), dtype=torch.float64, device="cuda")
        blocks = got["volts"].view(nt, nbin, nf)
        for i in range(nbin):
            power += torch.fft.fft(blocks[:, i].to(torch.complex128), dim=1).abs().square()
        return power.roll(nf // 2, dims=1).t().contiguous()
    band, dtype = (case["f_min"], case["f_max"]), case["dtype"]
    if kind == "batch":
        return [_like(_transform64(x, band, nd), dtype) for x, (_, _, nd) in zip(got["x"], _beams(case))]
    if kind == "stream":
        whole = _like(_transform64(torch.cat(got["x"], dim=1), band, case["nd"]), dtype)
        return [c.contiguous() for c in whole.split(case["chunk"], dim=1)]
    x = _mapped(got["x"], case)
    if kind == "step":
        w = got["w"].double()[:, None]
        back = _adjoint64(got["g"], band, case["nf"])
        return {"out": _transform64(x.double() * w, band, case["nd"]), "grad_x": _unmapped(back * w, case),
                "grad_w": (back * x.double()).sum(dim=1)}
    out = _transform64(x, band, case["nd"])
    if kind == "beam":
        return _like(out, dtype)
    sums, peaks = out, []
    for k in range(case["widths"]):
        if k:
            h = 1 << (k - 1)
            wider = sums.clone()
            wider[:, h:] += sums[:, :-h]
            sums = wider
        peaks.append(sums.amax(dim=1))
    peak = torch.stack(peaks, dim=1)
    # (equal peaks of rounded sums may come first at another time than exact ones)
    return {"out": _like(out, dtype), "peak": peak.round().to(torch.int64) if dtype == "u8" else peak, "time": None}
