"""The work whose speed counts: what users of the correlator X-engine have it do.

Every case is one pass through the package's public entry points on blocks that
are already on the device.  The kinds, each a use of the paper's X-engine:

  correlate  one whole integration in one call, from a few channels of the
             Pathfinder (256 inputs) to a band of full CHIME (2048 inputs)
  stream     an integration pushed block by block as the blocks arrive, and
             dumped (Sec. IV-C-1); short blocks, as the streaming service gets
  gated      pulsar gating (Sec. IV-C-4) with flagged samples (Sec. IV-A)
  shifted    time shifting (Sec. IV-C-5): a few inputs of an outlying station
             delayed, the history carried from push to push
  beams      beamforming (Sec. IV-C-3) at full sample cadence
  batch      independent integrations of uneven sizes, planned once

Results are whole numbers and have to be the same bits.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1503_06202_gb300 as xe

# Gates are phase bins of a pulse period; samples outside the bins are dropped.
GATE_DUTY = 0.95
# Operations that exact() takes on in 64 bits (about 1 T operations a second).
EXACT_OPS = 4e12


def listed():
    return [
        # the smallest call: eight channels of the Pathfinder, 10 ms of data
        {"name": "small", "kind": "correlate", "N": 256, "F": 8, "T": 4096, "sky": False},
        # the Pathfinder's full band, 84 ms of data: its real-time load
        {"name": "pathfinder", "kind": "correlate", "N": 256, "F": 1024, "T": 32768, "sky": True},
        # an array between the two telescopes, an odd number of 128-input blocks
        {"name": "mid", "kind": "correlate", "N": 640, "F": 128, "T": 8192, "sky": True},
        # a quarter of full CHIME's channels
        {"name": "chime", "kind": "correlate", "N": 2048, "F": 256, "T": 8192, "sky": True},
        # a node that holds four channels of the band and all the inputs
        {"name": "narrow", "kind": "correlate", "N": 1024, "F": 4, "T": 32768, "sky": True},
        # inputs and samples that fit no tile, no vector load
        {"name": "ragged", "kind": "correlate", "N": 203, "F": 64, "T": 10007, "sky": True},
        # short blocks of 0.66 ms integrated as they arrive
        {"name": "stream", "kind": "stream", "N": 512, "F": 256, "block": 256, "blocks": 8},
        # on and off pulse, 1% of the samples flagged
        {"name": "gated", "kind": "gated", "N": 256, "F": 256, "T": 16384, "gates": 2, "period": 128, "flags": True},
        # two inputs of an outlying station, 168 ms early
        {"name": "shifted", "kind": "shifted", "N": 1024, "F": 64, "T": 8192, "delayed": 2, "delay": 65625},
        # beams of full CHIME and of the Pathfinder
        {"name": "beams", "kind": "beams", "N": 2048, "F": 256, "T": 4096, "B": 16},
        {"name": "beams_narrow", "kind": "beams", "N": 256, "F": 128, "T": 16384, "B": 32},
        # 32 integrations of uneven sizes
        {"name": "batch", "kind": "batch", "jobs": 32, "sizes": 3, "n_max": 2048, "f_max": 64, "t_max": 32768},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _inputs(rng, lo, hi):
    """A number of inputs: a multiple of 16 twice in three (feeds come in boards of 16), else any."""
    n = _log(rng, lo, hi)
    return max(16, (n + 8) // 16 * 16) if rng.random() < 2 / 3 else n


def _draw(rng):
    kind = rng.choice(["correlate", "correlate", "stream", "gated", "shifted", "beams", "batch"])
    if kind == "correlate":
        return {"kind": kind, "N": _inputs(rng, 8, 2048), "F": _log(rng, 1, 1024), "T": _log(rng, 256, 65536),
                "sky": rng.random() < 0.75}
    if kind == "stream":
        return {"kind": kind, "N": _inputs(rng, 16, 2048), "F": _log(rng, 1, 512),
                "block": rng.choice([128, 256, 512, 1024, 200, _log(rng, 64, 2048)]), "blocks": rng.randint(2, 12)}
    if kind == "gated":
        return {"kind": kind, "N": _inputs(rng, 16, 2048), "F": _log(rng, 1, 512), "T": _log(rng, 512, 65536),
                "gates": rng.randint(1, 8), "period": _log(rng, 40, 4000), "flags": rng.random() < 0.7}
    if kind == "shifted":
        n = _inputs(rng, 16, 2048)
        return {"kind": kind, "N": n, "F": _log(rng, 1, 512), "T": _log(rng, 512, 32768),
                "delayed": rng.randint(1, min(16, n - 1)), "delay": _log(rng, 1, 100000)}
    if kind == "beams":
        return {"kind": kind, "N": 16 * _log(rng, 1, 128), "F": _log(rng, 1, 1024), "T": _log(rng, 256, 32768),
                "B": _log(rng, 1, 64)}
    return {"kind": kind, "jobs": rng.randint(4, 32), "sizes": rng.randrange(1 << 20), "n_max": 16 * _log(rng, 8, 128),
            "f_max": _log(rng, 2, 64), "t_max": _log(rng, 1024, 32768)}


def draw(rng):
    """One more case, of the listed ones' ranges and no dearer than the largest of them."""
    while True:
        case = _draw(rng)
        w = work(case)
        held = w["bytes"]
        if case["kind"] == "stream":  # every push reads and writes the triangle
            held += 16 * case["blocks"] * case["F"] * _pairs(case["N"])
        elif case["kind"] == "shifted":
            held += 2 * case["delay"] * case["F"] * case["delayed"]
        # what is neither a launch's latency nor dearer than a quarter of full CHIME
        if 1e6 <= w["bytes"] and held <= 4e9 and w["flops"] <= 1.5e13:
            return case


def _pairs(n):
    return n * (n + 1) // 2


def _batch_sizes(case):
    """(N, F, T) of a batch's jobs, from the case alone."""
    rng = random.Random(case["sizes"])
    ns = [n for n in (64, 96, 128, 200, 256, 512, 1024, 2048) if n <= case["n_max"]] + [case["n_max"]]
    fs = [f for f in (1, 16, 64) if f <= case["f_max"]] + [case["f_max"]]
    return [(rng.choice(ns), rng.choice(fs), 256 * max(1, _log(rng, 1024, case["t_max"]) // 256))
            for _ in range(case["jobs"])]


def _samples(case):
    return case["block"] * case["blocks"] if case["kind"] == "stream" else case["T"]


def work(case):
    """Bytes in and out once; 8 operations a complex multiply-accumulate."""
    if case["kind"] == "batch":
        sizes = _batch_sizes(case)
        return {"bytes": sum(t * f * n + 8 * f * _pairs(n) for n, f, t in sizes),
                "flops": 8 * sum(t * f * _pairs(n) for n, f, t in sizes)}
    n, f, t = case["N"], case["F"], _samples(case)
    if case["kind"] == "beams":
        b = case["B"]
        return {"bytes": t * f * n + 8 * t * f * b + 2 * f * b * n, "flops": 8 * t * f * b * n}
    out = 8 * f * _pairs(n)
    if case["kind"] == "gated":
        g = case["gates"]
        return {"bytes": t * f * n * (2 if case["flags"] else 1) + g * (out + 4 * f * n) + 4 * t,
                "flops": 8 * GATE_DUTY * t * f * _pairs(n)}
    if case["kind"] == "shifted":  # the history of the delayed inputs is read and written once
        return {"bytes": t * f * n + out + 2 * min(t, case["delay"]) * f * case["delayed"], "flops": 8 * t * f * _pairs(n)}
    return {"bytes": t * f * n + out, "flops": 8 * t * f * _pairs(n)}


def tolerance(case):
    return "exact"


def _generator(seed, device="cuda"):
    g = torch.Generator(device=device)
    g.manual_seed(seed)
    return g


def _block(T, F, N, sky, g):
    """uint8 [T][F][N]: two nibbles a sample, each value + 8.  sky: a signal that the
    inputs share (power 0.1) and receiver noise, rms 2.5; else uniform nibbles."""
    if not sky:
        return torch.randint(0, 256, (T, F, N), dtype=torch.uint8, device="cuda", generator=g)
    block = torch.empty((T, F, N), dtype=torch.uint8, device="cuda")
    step = max(1, (1 << 26) // (F * N))
    for t in range(0, T, step):
        n = min(step, T - t)
        x = torch.randn((2, n, F, N), device="cuda", generator=g)
        x.mul_(2.5 * math.sqrt(0.9)).add_(torch.randn((2, n, F, 1), device="cuda", generator=g), alpha=2.5 * math.sqrt(0.1))
        x = x.round_().clamp_(-8, 7).add_(8)
        block[t:t + n] = (16 * x[0] + x[1]).to(torch.uint8)
    return block


def _gate_list(case, seed):
    """int32 [T] on the host: the phase bin of each sample, -1 outside the bins."""
    rng = random.Random(seed)
    phase = ((np.arange(case["T"]) + rng.randrange(case["period"])) % case["period"]) / case["period"]
    gate = np.floor(phase / GATE_DUTY * case["gates"]).astype(np.int32)
    gate[gate >= case["gates"]] = -1
    return gate


def _delay_list(case, seed):
    """int32 [N]: the station's inputs, spread over the array, and their delays."""
    rng = random.Random(seed)
    delays = np.zeros(case["N"], np.int32)
    for i in rng.sample(range(case["N"]), case["delayed"]):
        delays[i] = max(1, case["delay"] - rng.randrange(1 + case["delay"] // 8))
    return delays


def _triangle(F, N, *lead):
    return torch.empty(lead + (F, _pairs(N), 2), dtype=torch.int32, device="cuda")


def prepare(case, seed):
    g = _generator(seed)
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "batch":
        s["jobs"] = [(_block(t, f, n, False, g), _triangle(f, n)) for n, f, t in _batch_sizes(case)]
        s["plan"] = xe.XBatch(s["jobs"])
        return s
    N, F = case["N"], case["F"]
    if kind == "beams":
        B = case["B"]
        s["block"] = _block(case["T"], F, N, True, g)
        s["weights"] = torch.randint(-128, 128, (2, F, B, N), dtype=torch.int8, device="cuda", generator=g)
        s["beam"] = xe.XBeam(N, F, B)
        s["beam"].set_weights(s["weights"][0], s["weights"][1])
        s["out"] = torch.empty((case["T"], F, B, 2), dtype=torch.int32, device="cuda")
        return s
    T = _samples(case)
    s["engine"] = xe.XEngine(N, F, T)
    s["out"] = _triangle(F, N)
    if kind == "stream":
        s["blocks"] = [_block(case["block"], F, N, True, g) for _ in range(case["blocks"])]
        return s
    s["block"] = _block(T, F, N, case.get("sky", True), g)
    if kind == "gated":
        s["gate"] = _gate_list(case, seed)
        s["valid"] = None
        if case["flags"]:
            s["valid"] = (torch.randint(0, 100, (T, F, N), dtype=torch.uint8, device="cuda", generator=g) > 0).to(torch.uint8)
        if xe.xeng_set_gates(s["engine"].h, case["gates"]) != xe.XENG_OK:
            raise RuntimeError("no memory for the gates")
        s["out"] = _triangle(F, N, case["gates"])
        s["counts"] = torch.empty((case["gates"], F, N), dtype=torch.int32, device="cuda")
    elif kind == "shifted":
        s["delays"] = _delay_list(case, seed)
        s["engine"].set_delays(s["delays"])
        # the stream so far: the history holds real samples
        s["engine"].push(s["block"])
        s["engine"].dump(s["out"])
        s["pushes"] = 1
    return s


def run(s):
    kind = s["kind"]
    if kind == "batch":
        s["plan"].run()
        return [out for _, out in s["jobs"]]
    if kind == "beams":
        s["beam"].run(s["block"], s["out"])
        return s["out"]
    eng = s["engine"]
    if kind == "correlate":
        eng.correlate(s["block"], s["out"])
        return s["out"]
    if kind == "gated":
        for rc in (xe.xeng_push_gated(eng.h, s["block"], s["block"].shape[0], s["gate"], s["valid"]),
                   xe.xeng_dump_gated(eng.h, s["out"], s["counts"])):
            if rc < 0:
                raise RuntimeError(xe.xeng_strerror(rc))
        return {"visibilities": s["out"], "counts": s["counts"]}
    for block in s["blocks"] if kind == "stream" else [s["block"]]:
        eng.push(block)
    eng.dump(s["out"])
    return s["out"]


def _complex(block):
    """The samples as (Re, Im) in 64 bits."""
    x = block.to(torch.int16)
    return (x >> 4).double() - 8, (x & 15).double() - 8


def _visibilities(re, im):
    """[F][pairs][2] of samples [T][F][N] in 64 bits: V_ij = sum x_i conj(x_j), i <= j."""
    T, F, N = re.shape
    upper = torch.triu_indices(N, N, device=re.device)
    out = torch.empty((F, _pairs(N), 2), dtype=torch.float64, device=re.device)
    for f in range(F):
        a, b = re[:, f].contiguous(), im[:, f].contiguous()
        v = a.T @ a + b.T @ b
        out[f, :, 0] = v[upper[0], upper[1]]
        v = b.T @ a
        out[f, :, 1] = (v - v.T)[upper[0], upper[1]]
    return out


def exact(case, seed):
    if work(case)["flops"] > EXACT_OPS or work(case)["bytes"] > 1.5e9:
        return None
    s = prepare(case, seed)
    kind = case["kind"]
    if kind == "batch":
        return [_visibilities(*_complex(block)) for block, _ in s["jobs"]]
    if kind == "stream":
        return _visibilities(*_complex(torch.cat(s["blocks"])))
    re, im = _complex(s["block"])
    if kind == "correlate":
        return _visibilities(re, im)
    if kind == "beams":
        out = torch.empty(s["out"].shape, dtype=torch.float64, device="cuda")
        w = s["weights"].double()
        for f in range(case["F"]):
            out[:, f, :, 0] = re[:, f] @ w[0, f].T - im[:, f] @ w[1, f].T
            out[:, f, :, 1] = re[:, f] @ w[1, f].T + im[:, f] @ w[0, f].T
        return out
    if kind == "gated":
        usable = torch.ones_like(re) if s["valid"] is None else s["valid"].double()
        gate = torch.from_numpy(s["gate"]).cuda()
        sets = [(gate == g).nonzero().flatten() for g in range(case["gates"])]
        return {"visibilities": torch.stack([_visibilities((re * usable)[t], (im * usable)[t]) for t in sets]),
                "counts": torch.stack([usable[t].sum(0) for t in sets])}
    # shifted: run()'s first pass is the stream's second push of the same block
    T = case["T"]
    for i in np.flatnonzero(s["delays"]):
        d = int(s["delays"][i])
        for x in (re, im):
            twice = torch.cat([torch.zeros((max(d - T, 0),) + x.shape[1:2], dtype=x.dtype, device=x.device), x[:, :, i], x[:, :, i]])
            x[:, :, i] = twice[len(twice) - T - d:len(twice) - d]
    return _visibilities(re, im)
