"""Performance cases: the calls that users of this library make, through its
public entry points, with the plans the library sets up by itself.

Every case dedisperses (or differentiates the dedispersion of) synthetic
observations: N(0, 1) noise plus a few dispersed pulses, in the input type
that the case names. 8-bit input has mean 128 and standard deviation 16, and
takes integer (Q8) weights. `weights` is "ones", or "masked": U(0.5, 1.5) with
one channel in twenty set to 0, as after the excision of interference.

  execute  Plan.execute on device tensors: an offline search, or one step of a
           pipeline whose data is on the GPU
  host     Plan.execute_host from and to pinned host memory: the whole call of
           a program that reads its data from a receiver or a file
  stream   a Stream reset and fed one observation in chunks: a real-time search
  learn    dedisperse and its gradients: learning the channel weights
  batch    Batch.execute: beams of two observation setups in one launch
"""
import math

import numpy as np
import torch

from paper_1601_05052_gb300 import Batch, Plan, Stream, dedisperse

# band: (lowest channel MHz, band top MHz, sampling time s, trial DM step)
BANDS = {
    "lband": (1400.0, 1500.0, 64e-6, 0.5),        # small L-band backend
    "apertif": (1420.0, 1720.0, 50e-6, 0.25),     # the paper's first setup
    "wide": (1250.0, 1550.0, 100e-6, 0.25),       # 300 MHz L-band receiver
    "lowfreq": (120.0, 180.0, 204.8e-6, 0.05),    # low-frequency tied-array beams
    "lofar": (138.0, 144.25, 5e-6, 0.25),         # the paper's second setup
}
TYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16, "u8": torch.uint8}


def _case(name, call, band, beams, chan, dm, out, dtype="f32", weights="ones", **more):
    c = {"call": call, "band": band, "beams": beams, "chan": chan, "dm": dm, "out": out,
         "dtype": dtype, "weights": weights}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one beam of a small backend, as a real-time loop calls it block by block: latency counts
        _case("beam_64ch_f32", "execute", "lband", 1, 64, 64, 4096),
        # the same with 8-bit input as it comes from the digitiser, masked channels
        _case("beam_64ch_u8", "execute", "lband", 1, 64, 64, 4096, "u8", "masked"),
        # 96 beams of that backend at once
        _case("beams96_64ch_f32", "execute", "lband", 96, 64, 64, 4096),
        # a handful of trials around a known DM over many beams: the memory-bound end
        _case("beams384_4dm_f32", "execute", "lband", 384, 64, 4, 4096),
        # survey scale, the paper's Apertif setup: one second, 2048 trial DMs
        _case("survey_f32", "execute", "apertif", 1, 1024, 2048, 20000),
        # the same from 8-bit data
        _case("survey_u8", "execute", "apertif", 1, 1024, 2048, 20000, "u8", "masked"),
        # two beams with a band edge cut off, sizes as they fall: half precision input
        _case("ragged_f16", "execute", "wide", 2, 509, 777, 10001, "f16", "masked"),
        # the paper's LOFAR setup: delays of neighbouring trials lie hundreds of samples apart
        _case("lofar_f32", "execute", "lofar", 1, 32, 2048, 200000),
        # survey scale from and to pinned host memory
        _case("survey_host_f32", "host", "apertif", 1, 1024, 2048, 20000),
        # real-time search: 4 chunks of 0.4 s, bfloat16 samples
        _case("stream_bf16", "stream", "wide", 1, 512, 1024, 4096, "bf16", "masked", chunks=4),
        # learning per-channel weights from 16 beams: forward, input and weight gradients
        _case("learn_f32", "learn", "wide", 16, 512, 1024, 8192),
        # beams of two receivers in one launch
        _case("batch_u8", "batch", "lband", 96, 64, 64, 4096, "u8",
              band2="lowfreq", beams2=32, chan2=256, dm2=2000, out2=10000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _adds(c):
    n = c["beams"] * c["chan"] * c["dm"] * c["out"] * c.get("chunks", 1)
    if c["call"] == "batch":
        n += c["beams2"] * c["chan2"] * c["dm2"] * c["out2"]
    return n * (3 if c["call"] == "learn" else 1)


def draw(rng):
    top = {c["call"]: 0 for c in listed()}
    for c in listed():
        top[c["call"]] = max(top[c["call"]], _adds(c))
    while True:
        call = rng.choice(["execute", "execute", "execute", "execute", "execute", "host", "stream",
                           "learn", "batch"])
        dtype = rng.choice(["f32", "f32", "f16", "bf16", "u8"])
        weights = rng.choice(["ones", "masked"])
        band = rng.choice(["lband", "lband", "apertif", "wide", "lowfreq", "lofar"])
        if call in ("learn", "stream", "host"):
            band = rng.choice(["lband", "apertif", "wide"])
        beams, chan, dm, out = {
            "lband": (_log(rng, 1, 384), _log(rng, 32, 128), _log(rng, 4, 128),
                      _log(rng, 1000, 8192)),
            "apertif": (_log(rng, 1, 4), _log(rng, 256, 1024), _log(rng, 64, 2048),
                        _log(rng, 4096, 20000)),
            "wide": (_log(rng, 1, 16), _log(rng, 128, 512), _log(rng, 64, 1024),
                     _log(rng, 2048, 10001)),
            "lowfreq": (_log(rng, 1, 32), _log(rng, 64, 256), _log(rng, 64, 2000),
                        _log(rng, 2048, 10000)),
            "lofar": (1, rng.choice([16, 31, 32]), _log(rng, 32, 2048), _log(rng, 20000, 200000)),
        }[band]
        c = _case("", call, band, beams, chan, dm, out, dtype, weights)
        if call == "learn":
            c["dtype"] = "f32"
        if call == "stream":
            c["chunks"] = rng.randint(2, 4)
        if call == "batch":
            c.update(band="lband", beams=_log(rng, 8, 96), chan=_log(rng, 32, 64),
                     dm=_log(rng, 16, 64), out=_log(rng, 1000, 4096), band2="lowfreq",
                     beams2=_log(rng, 2, 32), chan2=_log(rng, 64, 256), dm2=_log(rng, 200, 2000),
                     out2=_log(rng, 2048, 10000), dtype=rng.choice(["u8", "f16", "f32"]))
        if _adds(c) <= top[call] and work(c)["bytes"] <= 2.2e9:
            return c


def _setups(c):
    """The observation setups of a case (two for a batch)."""
    keys = ("band", "beams", "chan", "dm", "out")
    s = [tuple(c[k] for k in keys)]
    if c["call"] == "batch":
        s.append(tuple(c[k + "2"] for k in keys))
    return s


def _grid(band, chan, dm):
    """Channel frequencies, reference frequency, sampling time and trial DMs."""
    lo, hi, t_samp, step = BANDS[band]
    width = (hi - lo) / chan
    return lo + np.arange(chan) * width, hi - width, t_samp, np.arange(dm) * step


def _delays(band, chan, dm):
    """Delay table [dm][chan] in samples: Eq. 1 of the paper, halves away from zero."""
    f, f_ref, t_samp, dms = _grid(band, chan, dm)
    x = 4.148808e3 * dms[:, None] * (1.0 / (f * f) - 1.0 / (f_ref * f_ref))[None, :] / t_samp
    return np.floor(x + 0.5).astype(np.int64)


def _stride(t_in, dtype):
    n = 16 // TYPES[dtype].itemsize
    return -(-t_in // n) * n


def _inputs(c, setup, seed, n_beams=None):
    """(samples [beams][chan][stride], channel weights [chan]) on the GPU, from the seed."""
    band, beams, chan, dm, out = setup
    delays = _delays(band, chan, dm)
    length = out * c.get("chunks", 1) + (0 if c["call"] == "stream" else int(delays.max()))
    stride = length if c["call"] == "stream" else _stride(length, c["dtype"])
    gen = torch.Generator(device="cuda").manual_seed(seed * 1000003 + chan * 7919 + dm)
    x = torch.randn((beams, chan, stride), device="cuda", generator=gen)
    rng = np.random.default_rng(seed + 17)
    t = torch.arange(chan, device="cuda")
    for b in range(0, beams, max(1, beams // 10)):  # a pulse in some of the beams
        d, t0, amp = rng.integers(dm), rng.integers(out), rng.uniform(3, 10)
        at = torch.from_numpy(t0 + delays[d]).cuda()
        ok = at < length
        x[b, t[ok], at[ok]] += float(amp)
    w = torch.ones(chan, device="cuda")
    if c["weights"] == "masked":
        w = torch.empty(chan, device="cuda").uniform_(0.5, 1.5, generator=gen)
        w[torch.randperm(chan, device="cuda", generator=gen)[: (chan + 10) // 20]] = 0
    if c["dtype"] == "u8":
        x = x.mul_(16).add_(128).round_().clamp_(0, 255)
        w = torch.floor(256 * w + 0.5).to(torch.int32) if c["weights"] == "masked" else w.int()
    return x.to(TYPES[c["dtype"]]), w


def _plan(c, setup):
    band, beams, chan, dm, out = setup
    f, f_ref, t_samp, dms = _grid(band, chan, dm)
    return Plan(f, f_ref, t_samp, dms, out, batch=beams, dtype=c["dtype"])


def prepare(case, seed):
    plans = [_plan(case, s) for s in _setups(case)]
    data = [_inputs(case, s, seed) for s in _setups(case)]
    state = {"call": case["call"], "plan": plans[0], "x": data[0][0], "w": data[0][1]}
    if case["call"] == "host":
        state["x"] = state["x"].cpu().pin_memory()
        state["w"] = state["w"].cpu().pin_memory()
        state["out"] = torch.empty(plans[0].out_shape, dtype=plans[0].out_dtype).pin_memory()
    elif case["call"] == "stream":
        state["stream"] = Stream(plans[0])
        state["chunks"] = [k.contiguous() for k in data[0][0].split(case["out"], dim=2)]
    elif case["call"] == "learn":
        state["x"].requires_grad_(True)
        state["w"].requires_grad_(True)
        state["g"] = _cotangent(case, seed)
    elif case["call"] == "batch":
        state["batch"] = Batch(plans)
        state["x"], state["w"] = [d[0] for d in data], [d[1] for d in data]
    return state


def _cotangent(c, seed):
    """The gradient of a loss in a window of trials and samples, as it reaches the library."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 5)
    return torch.randn((c["beams"], c["dm"], c["out"]), device="cuda", generator=gen)


def run(state):
    call, plan = state["call"], state["plan"]
    if call == "execute":
        return plan.execute(state["x"], state["w"])
    if call == "host":
        return plan.execute_host(state["x"], state["w"], state["out"])
    if call == "stream":
        state["stream"].reset()
        return [state["stream"].push(k, state["w"]) for k in state["chunks"]]
    if call == "batch":
        return state["batch"].execute(state["x"], state["w"])
    out = dedisperse(plan, state["x"], state["w"])
    gx, gw = torch.autograd.grad(out, (state["x"], state["w"]), state["g"])
    return out.detach(), gx, gw


def work(case):
    """Bytes: each input sample, weight and output once. Flops: one add per
    channel and output, as the paper counts them (the gradients: one per
    channel and cotangent each)."""
    size = TYPES[case["dtype"]].itemsize
    total = flops = 0
    for band, beams, chan, dm, out in _setups(case):
        n = case.get("chunks", 1)
        span = 0 if case["call"] == "stream" else int(_delays(band, chan, dm).max())
        x, y = beams * chan * (out * n + span) * size, beams * dm * out * n * 4
        total += x + y + 4 * chan
        flops += beams * chan * dm * out * n
        if case["call"] == "learn":
            total += x + y + 4 * chan  # the cotangent in, the input and weight gradients out
            flops *= 3
    return {"bytes": total, "flops": flops}


def _shifted(rows, shifts, n):
    """[len(shifts)][n]: rows (1-D) from each shift on."""
    return rows.as_strided((rows.numel() - n + 1, n), (1, 1), rows.storage_offset())[shifts]


def exact(case, seed):
    if case["dtype"] == "u8":
        return None  # whole numbers: compared bit by bit
    band, beams, chan, dm, out = setup = _setups(case)[0]
    if case["call"] == "batch":
        return [_exact_forward(case, s, seed) for s in _setups(case)]
    if case["call"] == "stream":
        return _exact_stream(case, seed)
    y = _exact_forward(case, setup, seed)
    if case["call"] == "host":
        return y.cpu()
    if case["call"] != "learn":
        return y
    x, w = _inputs(case, setup, seed)
    g = _cotangent(case, seed)
    delays = _delays(band, chan, dm)
    span, length = int(delays.max()), x.shape[2]
    gx = torch.zeros(x.shape, dtype=torch.float64, device="cuda")
    gw = torch.zeros(chan, dtype=torch.float64, device="cuda")
    for b in range(beams):
        # g[d] behind `span` zeros: element tau + span - shift is g[d][tau - shift]
        pad = torch.zeros((dm, span + length), dtype=torch.float64, device="cuda")
        pad[:, span:span + out] = g[b].double()
        flat = pad.reshape(-1)
        row = torch.arange(dm, device="cuda") * (span + length)
        for c in range(chan):
            at = row + span - torch.from_numpy(delays[:, c]).cuda()
            sums = _shifted(flat, at, length).sum(0)
            gx[b, c] = sums * w[c].double()
            gw[c] += (sums * x[b, c].double()).sum()
    return y, gx, gw


def _exact_forward(case, setup, seed):
    band, beams, chan, dm, out = setup
    x, w = _inputs(case, setup, seed)
    delays = torch.from_numpy(_delays(band, chan, dm)).cuda()
    y = torch.zeros((beams, dm, out), dtype=torch.float64, device="cuda")
    for b in range(beams):
        for c in range(chan):
            y[b] += w[c].double() * _shifted(x[b, c].double(), delays[:, c], out)
    return y


def _exact_stream(case, seed):
    band, beams, chan, dm, out = setup = _setups(case)[0]
    x, w = _inputs(case, setup, seed)
    delays = torch.from_numpy(_delays(band, chan, dm)).cuda()
    span, n = int(delays.max()), out * case["chunks"]
    y = torch.zeros((beams, dm, n), dtype=torch.float64, device="cuda")
    for b in range(beams):
        for c in range(chan):
            row = torch.cat([torch.zeros(span, dtype=torch.float64, device="cuda"),
                             x[b, c].double()])
            y[b] += w[c].double() * _shifted(row, delays[:, c], n)
    return list(y.split(out, dim=2))
