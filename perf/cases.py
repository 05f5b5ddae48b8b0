"""The work a user of the correlator has it do, as cases that can be timed and checked.

A case is one X-stage call (or the few calls of one integration) through the public Python API:
samples that are already where the call wants them, a plan that the program keeps, and the
visibilities of one integration as the result.  ``listed()`` spans the range from a laboratory
array's smallest call to a 512-station block, over the three sample formats; ``draw()`` gives more
cases of the same kinds and ranges, odd sizes among them.

Kinds:

* ``dump``       one integration from device memory: ``Plan.execute_dump``;
* ``integrate``  one integration of 4- or 8-bit samples made of several executes, widened into int64
                 when it is dumped (the cross-dump sums): ``Plan.execute`` x n, ``Plan.dump(wide=True)``;
* ``batch``      uneven subarrays in one captured graph: ``Batch.replay``;
* ``host``       one integration from pinned host memory to pinned host memory:
                 ``Plan.execute_dump_host``.
"""

from __future__ import annotations

import math
import random

import torch

from paper_1401_8288_gb300 import xcorr

# The most that one drawn case may cost: complex multiply-adds of the integer formats and of the
# float format, and bytes moved (all at most those of the largest listed case).
MAX_CMACS = {"ci4": 1.37e11, "ci8": 1.37e11, "cf32": 0.7e11}
MAX_BYTES = 2.0e9
MAX_HOST_BYTES = 3.4e8
SAMPLE_BYTES = {"ci4": 1, "ci8": 2, "cf32": 8}


def _case(name, kind, fmt, n_sta, n_chan, n_time, **more):
    return {"name": name, "kind": kind, "fmt": fmt, "n_sta": n_sta, "n_chan": n_chan, "n_time": n_time, **more}


def listed():
    return [
        # the smallest call: one board of a laboratory array (8 stations, 16 channels), where the
        # host path and the launch are most of the time
        _case("ci4_16in_16ch_256t", "dump", "ci4", 8, 16, 256, keep_out=True),
        # a 32-station array, one short integration
        _case("ci4_64in_64ch_1024t", "dump", "ci4", 32, 64, 1024, keep_out=True),
        # a medium array; the caller lets the plan make the output
        _case("ci4_256in_256ch_1024t", "dump", "ci4", 128, 256, 1024, keep_out=False),
        # a large array's band on one GPU: the headline workload
        _case("ci4_512in_512ch_2048t", "dump", "ci4", 256, 512, 2048, keep_out=True),
        # a 512-station array's blocks added up over three executes and folded into wide sums
        _case("ci4_1024in_64ch_3x1024t_wide", "integrate", "ci4", 512, 64, 1024, executes=3),
        # an input count that is no multiple of 16, channels and samples that fill no tile
        _case("ci4_338in_97ch_1500t", "dump", "ci4", 169, 97, 1500, keep_out=False),
        # 8-bit samples of a 64-station array
        _case("ci8_128in_64ch_1024t", "dump", "ci8", 64, 64, 1024, keep_out=True),
        # 8-bit samples of a large array
        _case("ci8_512in_256ch_4096t", "dump", "ci8", 256, 256, 4096, keep_out=True),
        # float spectra of a GPU F-stage, a 64-station array
        _case("cf32_128in_64ch_1024t", "dump", "cf32", 64, 64, 1024, keep_out=False),
        # float spectra of a large array
        _case("cf32_512in_256ch_4096t", "dump", "cf32", 256, 256, 4096, keep_out=True),
        # 24 subarrays of uneven size sharing the GPU, replayed from one graph
        _case("batch_24_subarrays", "batch", "ci4", 0, 0, 0, count=24, max_sta=128, max_chan=256, max_time=4096,
              mix=7),
        # samples and visibilities in host memory (a capture process without device buffers)
        _case("host_ci4_512in_128ch_1024t", "host", "ci4", 256, 128, 1024),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dump", "dump", "dump", "dump", "dump", "dump", "integrate", "batch", "host"])
    if kind == "batch":
        return {"kind": "batch", "fmt": "ci4", "n_sta": 0, "n_chan": 0, "n_time": 0, "count": rng.randint(4, 32),
                "max_sta": _log_int(rng, 16, 128), "max_chan": _log_int(rng, 32, 256),
                "max_time": _log_int(rng, 512, 4096), "mix": rng.randint(0, 1 << 30)}
    fmt = rng.choice({"host": ["ci4"], "integrate": ["ci4", "ci8"]}.get(kind, ["ci4", "ci4", "ci8", "cf32"]))
    while True:
        n_sta = _log_int(rng, 8, 512)
        if rng.random() < 0.5 and n_sta >= 16:
            n_sta -= n_sta % 8  # half of the arrays have whole boards of 8 stations
        case = {"kind": kind, "fmt": fmt, "n_sta": n_sta, "n_chan": _log_int(rng, 16, 512),
                "n_time": _log_int(rng, 256, 4096)}
        if kind == "integrate":
            case["executes"] = rng.randint(2, 4)
        elif kind == "dump":
            case["keep_out"] = rng.random() < 0.5
        w = work(case)
        if w["flops"] / 8 <= MAX_CMACS[fmt] and w["bytes"] <= (MAX_HOST_BYTES if kind == "host" else MAX_BYTES):
            return case


def _subarrays(case):
    """(stations, channels, samples) of each subarray of a batch: stations in eights."""
    r = random.Random(case["mix"])
    return [(8 * max(1, _log_int(r, 8, case["max_sta"]) // 8), _log_int(r, 16, case["max_chan"]),
             _log_int(r, 256, case["max_time"])) for _ in range(case["count"])]


def _shapes(case):
    if case["kind"] == "batch":
        return _subarrays(case)
    return [(case["n_sta"], case["n_chan"], case["n_time"])] * case.get("executes", 1)


def work(case):
    nbytes = flops = 0
    elem = SAMPLE_BYTES[case["fmt"]]
    for k, (s, c, t) in enumerate(_shapes(case)):
        pairs = s * (2 * s + 1)
        nbytes += elem * t * c * 2 * s
        flops += 8 * t * c * pairs
        if case["kind"] == "integrate":
            nbytes += 16 * c * pairs if k == 0 else 0  # int64 sums, written once
        else:
            nbytes += 8 * c * pairs
    return {"bytes": nbytes, "flops": flops}


def _samples(fmt, n_sta, n_chan, n_time, gen):
    """Receiver noise plus one weak common source (0.3 of the noise, a phase per channel and input)."""
    n_in = 2 * n_sta
    shape = {"ci4": (n_time, n_chan, n_sta, 2), "ci8": (n_time, n_chan, n_sta, 2, 2),
             "cf32": (n_time, n_chan, n_sta, 2, 2)}[fmt]
    out = torch.empty(shape, dtype={"ci4": torch.uint8, "ci8": torch.int8, "cf32": torch.float32}[fmt], device="cuda")
    turn = torch.rand((n_chan, n_in), generator=gen, device="cuda") * (2 * math.pi)
    cos, sin = 0.3 * turn.cos(), 0.3 * turn.sin()
    sigma, top = {"ci4": (2.5, 7), "ci8": (20.0, 127), "cf32": (1.0, 0)}[fmt]
    step = max(1, (1 << 25) // (n_chan * n_in))
    for t0 in range(0, n_time, step):
        n = min(step, n_time - t0)
        s = torch.randn((2, n, n_chan, 1), generator=gen, device="cuda")
        re = torch.randn((n, n_chan, n_in), generator=gen, device="cuda").addcmul_(s[0], cos).addcmul_(s[1], -sin)
        im = torch.randn((n, n_chan, n_in), generator=gen, device="cuda").addcmul_(s[0], sin).addcmul_(s[1], cos)
        re, im = re.mul_(sigma), im.mul_(sigma)
        if top:
            re, im = re.round_().clamp_(-top, top).to(torch.int8), im.round_().clamp_(-top, top).to(torch.int8)
        if fmt == "ci4":
            v = ((re << 4) | (im & 15)).view(torch.uint8)
        else:
            v = torch.stack((re, im), dim=-1)
        out[t0:t0 + n] = v.reshape((n,) + shape[1:])
    return out


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(0x14018288 + int(seed))
    return [_samples(case["fmt"], s, c, t, gen) for s, c, t in _shapes(case)]


def prepare(case, seed):
    xs = _inputs(case, seed)
    if case["kind"] == "batch":
        batch = xcorr.Batch(_subarrays(case))
        batch.capture(xs)
        return {"kind": "batch", "batch": batch, "x": xs}
    s, c, t = case["n_sta"], case["n_chan"], case["n_time"]
    plan = xcorr.Plan(s, c, t, fmt=case["fmt"])
    state = {"kind": case["kind"], "plan": plan, "x": xs, "out": None}
    shape, dtype = (c, s * (2 * s + 1), 2), torch.float32 if case["fmt"] == "cf32" else torch.int32
    if case["kind"] == "host":
        state["x"] = [xs[0].cpu().pin_memory()]
        state["out"] = torch.empty(shape, dtype=dtype, pin_memory=True)
    elif case.get("keep_out"):
        state["out"] = torch.empty(shape, dtype=dtype, device="cuda")
    return state


def run(state):
    kind, xs = state["kind"], state["x"]
    if kind == "batch":
        return list(state["batch"].replay())
    plan = state["plan"]
    if kind == "dump":
        return plan.execute_dump(xs[0], out=state["out"])
    if kind == "integrate":
        for x in xs:
            plan.execute(x)
        return plan.dump(wide=True)
    out = plan.execute_dump_host(xs[0], out=state["out"])
    plan.sync()  # the visibilities are in host memory after this
    return out


def _visibilities(fmt, x):
    """sum_t x x^H of one [t][c][s][2] input in FP64, the packed lower triangle [c][pair][2]."""
    n_time, n_chan = x.shape[:2]
    n_in = x.shape[2] * 2
    row, col = torch.tril_indices(n_in, n_in, device="cuda")
    out = torch.empty((n_chan, row.numel(), 2), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 26) // (n_time * n_in))
    for c0 in range(0, n_chan, step):
        v = x[:, c0:c0 + step]
        n = v.shape[1]
        if fmt == "ci4":
            v = v.view(torch.int8)
            re, im = v >> 4, (v << 4) >> 4
        else:
            re, im = v[..., 0], v[..., 1]
        re = re.reshape(n_time, n, n_in).permute(1, 2, 0).to(torch.float64)
        im = im.reshape(n_time, n, n_in).permute(1, 2, 0).to(torch.float64)
        rt, it = re.transpose(1, 2), im.transpose(1, 2)
        out[c0:c0 + n, :, 0] = (re @ rt + im @ it)[:, row, col]
        m = im @ rt
        out[c0:c0 + n, :, 1] = (m - m.transpose(1, 2))[:, row, col]
    return out


def exact(case, seed):
    if work(case)["flops"] > 3e12:  # FP64 matrix products of this size take too long
        return None
    xs = _inputs(case, seed)
    vs = []
    for x in xs:
        vs.append(_visibilities(case["fmt"], x))
    if case["kind"] == "integrate":
        vs = [sum(vs[1:], vs[0])]
    if case["fmt"] != "cf32":
        vs = [v.to(torch.int64) for v in vs]
    return vs if case["kind"] == "batch" else vs[0].cpu() if case["kind"] == "host" else vs[0]
