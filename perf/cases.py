"""The work a user of this library has it do, as cases that can be timed and checked.

Every case goes through the public Python entry points (``Plan``, ``Batch``, ``MultiRatePlan``,
``Sifter``, ``snippets``). The streaming calls are timed in the steady state of a stream: the
filterbank of a case is periodic (noise with dispersed bursts whose sweeps wrap round its
end), the delay history is filled by ``prepare``, and every ``run`` takes the stream's next
chunk and reads the candidates, as a search loop does.

Kinds of call:
  stream     Plan.execute (a chunk on the device) or Plan.execute_host (a chunk in pinned host
             memory) and Plan.candidates; plane: "none" (a search keeps the candidates only),
             "full" (int32, or float32 in float mode and for the labelled payload) or "u8"
  batch      Batch.execute over ragged beams and every beam's candidates
  multirate  MultiRatePlan.execute and the merged candidates
  sift       snippets of a float plane around candidates, and the classifier's logits
  train      loss and gradients of one labelled batch (forward and backward)

``exact`` states the same definitions once more in plain torch in 64 bits (integer counts are
exact): encoder levels, node rules, boxcar S/N, closing, islands and peaks.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch
import torch.nn.functional as F

import paper_2606_15361_gb300 as snd

DT = 1.38e-4       # s
F_TOP, BW = 416.0, 16.0
K_DM = 4.148808e3  # MHz^2 s pc^-1 cm^3
WMAX = 1024        # widest boxcar
CAND_ROWS = 512    # rows a beam's candidate list is padded to
MODES = {"binary": snd.MODE_BINARY, "graded": snd.MODE_GRADED, "float": snd.MODE_FLOAT, "zfloat": snd.MODE_ZFLOAT}
THETA = {"binary": 1.5, "graded": 0.75, "float": 1.5, "zfloat": 1.5}  # encoder thresholds of the operating points


# ------------------------------------------------------------------------------- cases

def listed():
    return [
        # the smallest beam in short blocks, compact plane kept: latency of a low-delay search
        {"name": "nc64_binary_1k", "call": "stream", "mode": "binary", "nchan": 64, "ndm": 128, "dm_max": 100.0,
         "nsamp": 1024, "branching": 4, "host": False, "plane": "u8"},
        # the 64-channel beam in ordinary chunks, plane kept
        {"name": "nc64_float_plane", "call": "stream", "mode": "float", "nchan": 64, "ndm": 128, "dm_max": 100.0,
         "nsamp": 16384, "branching": 2, "host": False, "plane": "full"},
        # the Northern Cross beam in its three modes: candidates and the compact plane; candidates
        # only, chunks arriving in host memory; and the float plane that the sifter reads
        {"name": "nc1024_binary_u8", "call": "stream", "mode": "binary", "nchan": 1024, "ndm": 2048, "dm_max": 2000.0,
         "nsamp": 16384, "branching": 8, "host": False, "plane": "u8"},
        {"name": "nc1024_graded_host", "call": "stream", "mode": "graded", "nchan": 1024, "ndm": 2048,
         "dm_max": 2000.0, "nsamp": 16384, "branching": 8, "host": True, "plane": "none"},
        {"name": "nc1024_float_plane", "call": "stream", "mode": "float", "nchan": 1024, "ndm": 2048,
         "dm_max": 2000.0, "nsamp": 16384, "branching": 8, "host": False, "plane": "full"},
        # a band with flagged edges: channel count, DM count and chunk length with no round factors
        {"name": "nc1000_graded_ragged", "call": "stream", "mode": "graded", "nchan": 1000, "ndm": 1537,
         "dm_max": 1500.0, "nsamp": 10007, "branching": 8, "host": False, "plane": "none"},
        # finest channelisation, the highest DMs, one second a chunk
        {"name": "nc4096_float", "call": "stream", "mode": "float", "nchan": 4096, "ndm": 4096, "dm_max": 3000.0,
         "nsamp": 7246, "branching": 4, "host": False, "plane": "none"},
        # the precision study: labelled payload with FP16 partial sums
        {"name": "nc1024_zfloat_fp16", "call": "stream", "mode": "zfloat", "nchan": 1024, "ndm": 2048,
         "dm_max": 2000.0, "nsamp": 16384, "branching": 8, "host": False, "plane": "full", "fp16": True},
        # several beams of one receiver a step, each with its own DM grid and chunk length
        {"name": "beams8_float", "call": "batch", "mode": "float", "nchan": 1024, "beams": 8, "ndm_lo": 512,
         "ndm_hi": 4096, "dm_lo": 500.0, "dm_hi": 3000.0, "nsamp_lo": 4096, "nsamp_hi": 32768, "branching": 8,
         "shapes": 11},
        # the multi-rate search over the whole DM range
        {"name": "multirate_graded", "call": "multirate", "mode": "graded", "nchan": 1024, "ndm": 2048,
         "dm_max": 2000.0, "nsamp": 16384, "branching": 8, "s_max": 16},
        # learned sifter: a full inference batch from the plane, and a training batch
        {"name": "sift_4096", "call": "sift", "n": 4096, "ndm": 2048, "ncols": 16384},
        {"name": "train_256", "call": "train", "n": 256},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _root_fires(nchan, branching):
    """Whether a binary tree's root can reach its quorum of two (a ragged end can rule it out)."""
    ok = [min(4, nchan - c) >= 2 for c in range(0, nchan, 4)]
    while len(ok) > 1:
        ok = [sum(ok[i:i + branching]) >= 2 for i in range(0, len(ok), branching)]
    return ok[0]


def draw(rng):
    """One more case of the listed ranges."""
    kind = rng.choice(["stream", "stream", "stream", "stream", "zfloat", "batch", "multirate", "sift", "train"])
    if kind == "sift":
        return {"call": "sift", "n": _log_int(rng, 16, 4096), "ndm": _log_int(rng, 128, 2048),
                "ncols": _log_int(rng, 1024, 16384)}
    if kind == "train":
        return {"call": "train", "n": _log_int(rng, 32, 512)}
    mode = rng.choice(["binary", "graded", "float"])
    branching = rng.choice([4, 8] if mode == "binary" else [2, 4, 8])
    if kind == "batch":
        nchan = 64 * rng.choice([n for n in range(2, 17) if mode != "binary" or _root_fires(64 * n, branching)])
        return {"call": "batch", "mode": mode, "nchan": nchan, "beams": rng.randint(2, 8),
                "ndm_lo": 256, "ndm_hi": _log_int(rng, 512, 4096), "dm_lo": 300.0, "dm_hi": 2000.0,
                "nsamp_lo": 4096, "nsamp_hi": 16384, "branching": branching, "shapes": rng.randint(1, 10 ** 6)}
    # channel counts: blocks of 64, or any number (flagged channels)
    nchan = 64 * _log_int(rng, 1, 32) if rng.random() < 0.5 else _log_int(rng, 64, 2048)
    while mode == "binary" and not _root_fires(nchan, branching):
        nchan = _log_int(rng, 64, 2048)
    ndm = _log_int(rng, 100, 3000 if nchan > 1100 else 4096)
    # trial DMs as fine as the listed grids, so that the sweep between neighbours stays short
    dm_max = round(min(3000.0, ndm * rng.uniform(0.3, 1.0)), 1)
    nsamp = _log_int(rng, 700, 16384)
    if kind == "multirate":
        return {"call": "multirate", "mode": mode, "nchan": max(128, nchan), "ndm": max(ndm, 1000),
                "dm_max": max(dm_max, 800.0), "nsamp": 16 * _log_int(rng, 128, 1024), "branching": branching,
                "s_max": rng.choice([4, 8, 16])}
    if kind == "zfloat":
        return {"call": "stream", "mode": "zfloat", "nchan": min(nchan, 1024), "ndm": min(ndm, 2048), "dm_max": dm_max,
                "nsamp": nsamp, "branching": branching, "host": False, "plane": "full", "fp16": rng.random() < 0.5}
    plane = rng.choice(["none" if nsamp >= 2048 else "full", "full", "full" if mode == "float" else "u8"])
    return {"call": "stream", "mode": mode, "nchan": nchan, "ndm": ndm, "dm_max": dm_max, "nsamp": nsamp,
            "branching": branching, "host": rng.random() < 0.25, "plane": plane}


def work(case):
    """Inputs read once and outputs written once; additions of direct dedispersion and of the boxcar
    sums per DM-sample (the multi-rate search runs each DM at its own rate)."""
    call = case["call"]
    if call == "sift":
        n = case["n"]
        return {"bytes": 2 * n * 64 * 256 * 4 + 4 * n, "flops": n * _sifter_flops()}
    if call == "train":
        return {"bytes": case["n"] * (64 * 256 * 4 + 4) + 4 * _num_params(), "flops": 3 * case["n"] * _sifter_flops()}
    if call == "batch":
        b = f = 0
        for ndm, _, nsamp in _beam_shapes(case):
            b += nsamp * case["nchan"]
            f += float(ndm) * nsamp * (case["nchan"] + 10)
        return {"bytes": b, "flops": f}
    nchan, ndm, nsamp = case["nchan"], case["ndm"], case["nsamp"]
    if call == "multirate":
        scr = _scrunch(case)
        return {"bytes": nchan * nsamp, "flops": sum((nchan + 10.0) * nsamp / s for s in scr)}
    per = {"none": 0, "full": 4, "u8": 1}[case["plane"]]
    return {"bytes": nchan * nsamp + per * ndm * nsamp, "flops": float(ndm) * nsamp * (nchan + 10)}


# ------------------------------------------------------------------------------- inputs

def _freqs(nchan):
    return F_TOP - (np.arange(nchan, dtype=np.float64) + 0.5) * (BW / nchan)


def _sweep(nchan, dm):
    f = _freqs(nchan)
    return K_DM * dm * (f.min() ** -2 - f.max() ** -2) / DT


def _filterbank(nchan, nsamp, nchunks, dm_max, bright, seed):
    """Periodic filterbank uint8 [nchunks * nsamp][nchan] on the GPU: noise N(128, 16) and
    dispersed Gaussian bursts, 200 in 2^18 samples, FWHM 1-72 samples, S/N 6-50, one in every chunk
    short (FWHM 1-6) and of S/N `bright`."""
    total = nchunks * nsamp
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((total, nchan), generator=gen, device="cuda", dtype=torch.float32).mul_(16.0).add_(128.0)
    rng = random.Random(seed)
    f = torch.from_numpy(_freqs(nchan)).cuda()
    chan = torch.arange(nchan, device="cuda")[:, None]
    for i in range(max(nchunks, round(total * 200 / 2 ** 18))):
        t0 = rng.uniform(0, total) if i >= nchunks else (i + rng.random()) * nsamp
        dm = rng.uniform(0.01, 0.99) * dm_max
        sig = math.exp(rng.uniform(0.0, math.log(72.0 if i >= nchunks else 6.0))) / 2.3548
        snr = math.exp(rng.uniform(math.log(6.0), math.log(50.0))) if i >= nchunks else bright
        half = int(math.ceil(4.0 * sig)) + 1
        centre = t0 + K_DM * dm * (f ** -2 - f.max() ** -2) / DT
        tt = torch.floor(centre).long()[:, None] + torch.arange(-half, half + 1, device="cuda")
        prof = torch.exp(-0.5 * ((tt.double() - centre[:, None]) / sig) ** 2)
        amp = snr / math.sqrt(nchan * math.sqrt(math.pi) * sig)
        # every (sample, channel) comes once: a burst is shorter than the period
        x[tt % total, chan.expand_as(tt)] += (16.0 * amp * prof).float()
    return x.round_().clamp_(0, 255).to(torch.uint8)


def _history(case, wmax_native=WMAX):
    """Chunks that fill the stream (sweep and widest boxcar), and the period of the filterbank."""
    need = _sweep(case["nchan"], case["dm_max"]) + wmax_native + 2
    fill = int(math.ceil(need / case["nsamp"]))
    return fill, fill + 2


def _options(case):
    o = snd.options(MODES[case["mode"]], max_chunk=case["nsamp"])
    if case.get("plane") == "u8":
        o.plane_dtype = 1
    if case.get("fp16"):
        o.flags = snd.FLAG_FP16_PARTIALS
    return o


def _beam_shapes(case):
    """(DMs, largest DM, chunk length) of every beam, chunk lengths in steps of 1024."""
    rng = random.Random(case["shapes"])
    out = []
    for _ in range(case["beams"]):
        ndm = rng.randint(case["ndm_lo"], case["ndm_hi"])
        dm = min(rng.uniform(case["dm_lo"], case["dm_hi"]), 1.0 * ndm)
        out.append((ndm, round(dm, 1), 1024 * rng.randint(case["nsamp_lo"] // 1024, case["nsamp_hi"] // 1024)))
    return out


def _beam_case(case, i):
    ndm, dm, nsamp = _beam_shapes(case)[i]
    return {"call": "stream", "mode": case["mode"], "nchan": case["nchan"], "ndm": ndm, "dm_max": dm, "nsamp": nsamp,
            "branching": case["branching"], "plane": "none"}


def _sifter_flops():
    # two per multiply-add of the three convolutions and the two dense layers
    return 2 * (64 * 256 * 16 * 9 + 32 * 128 * 32 * 144 + 16 * 64 * 64 * 288 + 16384 * 128 + 128)


def _num_params():
    return 16 * 9 + 16 + 32 * 144 + 32 + 64 * 288 + 64 + 128 * 16384 + 128 + 128 + 1


def _params():
    """Weights of a classifier at the start of training (He-uniform, small biases), as one vector."""
    r = np.random.default_rng(7)
    parts = []
    for shape, fan in (((16, 1, 3, 3), 9), ((32, 16, 3, 3), 144), ((64, 32, 3, 3), 288), ((128, 16384), 16384),
                       ((128,), 128)):
        lim = math.sqrt(6.0 / fan)
        parts.append(r.uniform(-lim, lim, int(np.prod(shape))))
        parts.append(r.uniform(-0.05, 0.05, shape[0] if len(shape) > 1 else 1))
    return np.concatenate(parts).astype(np.float32)


def _plane(ndm, ncols, gen):
    """A float plane of noise: counts over 32, as the float mode writes for 1024 channels."""
    return torch.randn((ndm, ncols), generator=gen, device="cuda").mul_(8.0).add_(68.0).round_().div_(32.0)


def _snippet_batch(n, gen):
    """Standardised snippets, about half of them with a bow tie, and their labels."""
    x = torch.randn((n, 64, 256), generator=gen, device="cuda")
    y = (torch.rand(n, generator=gen, device="cuda") < 0.5).float()
    d = torch.arange(-32, 32, device="cuda", dtype=torch.float32)[:, None]
    t = torch.arange(-128, 128, device="cuda", dtype=torch.float32)[None, :]
    amp = torch.rand(n, generator=gen, device="cuda") * 6.0 + 2.0
    width = torch.rand(n, generator=gen, device="cuda") * 8.0 + 2.0
    sig = width[:, None, None] + d.abs()
    x += (amp * y)[:, None, None] * (width[:, None, None] / sig) * torch.exp(-0.5 * (t / sig) ** 2)
    x = (x - x.mean(dim=(1, 2), keepdim=True)) / x.std(dim=(1, 2), keepdim=True)
    return x.contiguous(), y


# ------------------------------------------------------------------------------- prepare and run

def prepare(case, seed):
    call = case["call"]
    if call == "sift":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        plane = _plane(case["ndm"], case["ncols"], gen)
        n = case["n"]
        rows = torch.randint(0, case["ndm"], (n,), generator=gen, device="cuda").int()
        cols = torch.randint(0, case["ncols"], (n,), generator=gen, device="cuda")
        sifter = snd.Sifter(n, training=False)
        sifter.set_params(_params())
        return {"call": call, "plane": plane, "rows": rows, "cols": cols, "sifter": sifter,
                "x": torch.empty((n, 64, 256), device="cuda"), "logits": torch.empty(n, device="cuda")}
    if call == "train":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        x, y = _snippet_batch(case["n"], gen)
        sifter = snd.Sifter(case["n"], training=True)
        sifter.set_params(_params())
        return {"call": call, "x": x, "y": y, "sifter": sifter}
    if call == "batch":
        plans, beams = [], []
        for i in range(case["beams"]):
            c = _beam_case(case, i)
            plans.append(_make_plan(c))
            beams.append(_stream_chunks(c, seed + 1000 * i))
        fill = max(b["fill"] for b in beams)
        batch = snd.Batch(plans)
        for k in range(fill):
            batch.execute([b["chunks"][k % len(b["chunks"])] for b in beams])
            if k % 8 == 7:
                [p.candidates(check=False) for p in plans]
        [p.candidates(check=False) for p in plans]
        return {"call": call, "plans": plans, "batch": batch, "beams": beams, "next": fill}
    if call == "multirate":
        b = _stream_chunks(case, seed, _multirate_reach(case))
        plan = snd.MultiRatePlan(_freqs(case["nchan"]), DT, np.linspace(0.0, case["dm_max"], case["ndm"]),
                                 case["branching"], MODES[case["mode"]], _options(case), s_max=case["s_max"])
        for k in range(b["fill"]):
            plan.execute(b["chunks"][k])
            if k % 8 == 7:
                plan.candidates(check=False)
        plan.candidates(check=False)
        return {"call": call, "plan": plan, "chunks": b["chunks"], "next": b["fill"]}
    b = _stream_chunks(case, seed)
    plan = _make_plan(case)
    for k in range(b["fill"]):
        plan.execute(b["chunks"][k])
        if k % 8 == 7:
            plan.candidates(check=False)
    plan.candidates(check=False)
    chunks = b["chunks"]
    if case["host"]:
        chunks = [c.cpu().pin_memory() for c in chunks]
    out = None
    if case["plane"] != "none":
        dtype = torch.uint8 if case["plane"] == "u8" else (
            torch.float32 if case["mode"] in ("float", "zfloat") else torch.int32)
        out = torch.empty((case["ndm"], case["nsamp"]), dtype=dtype, device="cuda")
    return {"call": call, "plan": plan, "chunks": chunks, "next": b["fill"], "host": case["host"], "out": out,
            "search": case["mode"] != "zfloat"}


def _make_plan(case):
    return snd.Plan(_freqs(case["nchan"]), DT, np.linspace(0.0, case["dm_max"], case["ndm"]), case["branching"],
                    MODES[case["mode"]], _options(case))


def _stream_chunks(case, seed, reach=WMAX):
    fill, nchunks = _history(case, reach)
    # a binary tree's quorums want a burst that shows in single channels
    bright = 4.0 * math.sqrt(case["nchan"]) if case["mode"] == "binary" else 40.0
    data = _filterbank(case["nchan"], case["nsamp"], nchunks, case["dm_max"], bright, seed)
    return {"fill": fill, "chunks": list(data.view(nchunks, case["nsamp"], case["nchan"]))}


def _columns(cands):
    """The candidate list as columns of a fixed length (rows past the list are zero)."""
    pad = np.zeros(CAND_ROWS, dtype=cands.dtype)
    n = min(len(cands), CAND_ROWS)
    pad[:n] = cands[:n]
    return {"n": len(cands), "dm_index": pad["dm_index"], "t": pad["t"], "snr": pad["snr"], "width": pad["width"],
            "npix": pad["npix"]}


def run(state):
    call = state["call"]
    if call == "sift":
        x = snd.snippets(state["plane"], state["rows"], state["cols"], out=state["x"])
        return {"x": x, "logits": state["sifter"].forward(x, state["logits"])}
    if call == "train":
        loss, grads = state["sifter"].gradients(state["x"], state["y"])
        return {"loss": loss, "grads": grads}
    k = state["next"]
    state["next"] = k + 1
    if call == "batch":
        state["batch"].execute([b["chunks"][k % len(b["chunks"])] for b in state["beams"]])
        return [_columns(p.candidates()[0]) for p in state["plans"]]
    plan, chunk = state["plan"], state["chunks"][k % len(state["chunks"])]
    if call == "multirate":
        plan.execute(chunk)
        return _columns(plan.candidates()[0])
    if state["host"]:
        plan.execute_host(chunk, state["out"])
    else:
        plan.execute(chunk, state["out"])
    if not state["search"]:
        return {"plane": state["out"]}
    out = _columns(plan.candidates()[0])
    if state["out"] is not None:
        out["plane"] = state["out"]
    return out


# ------------------------------------------------------------------------------- exact

def exact(case, seed):
    """The outputs of the first run on these inputs, in 64 bits; None in the place of whole
    numbers (they are compared as they are)."""
    call = case["call"]
    if call == "sift":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        plane = _plane(case["ndm"], case["ncols"], gen)
        n = case["n"]
        rows = torch.randint(0, case["ndm"], (n,), generator=gen, device="cuda").int()
        cols = torch.randint(0, case["ncols"], (n,), generator=gen, device="cuda")
        x = _exact_snippets(plane, rows.long(), cols)
        w = _split_params(torch.from_numpy(_params()).cuda().double())
        return {"x": x, "logits": torch.cat([_network(x[i:i + 128], w) for i in range(0, n, 128)])}
    if call == "train":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        x, y = _snippet_batch(case["n"], gen)
        p = torch.from_numpy(_params()).cuda().double().requires_grad_(True)
        loss = 0.0
        for i in range(0, case["n"], 64):
            z = _network(x[i:i + 64].double(), _split_params(p))
            part = F.binary_cross_entropy_with_logits(z, y[i:i + 64].double(), reduction="sum") / case["n"]
            part.backward()
            loss += float(part)
        return {"loss": torch.tensor([loss], dtype=torch.float64), "grads": p.grad}
    if call == "batch":
        out = []
        for i in range(case["beams"]):
            c = _beam_case(case, i)
            b = _stream_chunks(c, seed + 1000 * i)
            fill = max(_history(_beam_case(case, j))[0] for j in range(case["beams"]))
            out.append(_exact_columns(_search(c, b["chunks"], fill)[0]))
            del b
        return out
    if call == "multirate":
        chunks = _stream_chunks(case, seed, _multirate_reach(case))["chunks"]
        return _exact_columns(_exact_multirate(case, chunks))
    b = _stream_chunks(case, seed)
    if case["mode"] == "zfloat":
        return {"plane": _exact_zfloat(case, b["chunks"], b["fill"])}
    cands, plane = _search(case, b["chunks"], b["fill"])
    out = _exact_columns(cands)
    if case["plane"] != "none":
        out["plane"] = plane / math.sqrt(case["nchan"]) if case["mode"] == "float" else None
    return out


def _exact_columns(cands):
    snr = np.zeros(CAND_ROWS, dtype=np.float64)
    n = min(len(cands), CAND_ROWS)
    snr[:n] = [c[2] for c in cands[:n]]
    return {"n": None, "dm_index": None, "t": None, "snr": snr, "width": None, "npix": None}


def _delays(nchan, dt, dms):
    f = _freqs(nchan)
    inv2 = 1.0 / (f * f)
    return np.floor((K_DM * np.asarray(dms))[:, None] * (inv2 - inv2[0])[None, :] / dt + 0.5).astype(np.int64)


def _levels(chunk, theta):
    """Per channel: firing level (smallest firing value, 256: never), clipped mean and deviation."""
    nchan = chunk.shape[1]
    v = torch.arange(256, device=chunk.device, dtype=torch.float64)
    flat = (torch.arange(nchan, device=chunk.device)[None, :] * 256 + chunk.long()).reshape(-1)
    h = torch.bincount(flat, minlength=nchan * 256).view(nchan, 256).double()
    n = float(chunk.shape[0])
    mu0 = (h @ v) / n
    sig0 = ((h @ (v * v)) / n - mu0 ** 2).clamp_min(0).sqrt()
    c = torch.maximum(torch.minimum(v[None, :], (mu0 + 5 * sig0)[:, None]), (mu0 - 5 * sig0)[:, None])
    mu = (h * c).sum(1) / n
    sig = ((h * c * c).sum(1) / n - mu ** 2).clamp_min(0).sqrt()
    u = (torch.floor(mu + theta * sig) + 1).clamp(0, 256)
    return torch.where(sig > 0, u, torch.full_like(u, 256.0)), mu, sig


def _extended(series, total, reach):
    """[nchan][total] continued periodically to `reach` samples past its end."""
    reps = 1 + (reach + total - 1) // total
    return series.repeat(1, reps)


def _search(case, chunks, fill, dt=DT, dms=None):
    """(candidates [(t, dm index, snr64, width, npix)] of the chunk after `fill` chunks, its plane)."""
    mode, nchan, nsamp, branching = case["mode"], case["nchan"], chunks[0].shape[0], case["branching"]
    dms = np.linspace(0.0, case["dm_max"], case["ndm"]) if dms is None else dms
    delay = _delays(nchan, dt, dms)
    D, ndm = int(delay.max()), len(dms)
    sweep = (K_DM * dms) * (_freqs(nchan)[-1] ** -2 - _freqs(nchan)[0] ** -2) / dt
    widths = [[w for w in (1 << j for j in range(11)) if w <= 8 or w <= 0.1 * s] for s in sweep]
    wmax = max(w[-1] for w in widths)
    fired = torch.cat([(c.t() >= _levels(c, THETA[mode])[0][:, None]) for c in chunks], 1).to(torch.uint8)
    total = fired.shape[1]
    f0 = fill * nsamp - D - (wmax - 1)  # first start time of the block; E_prev = f0 + wmax - 1
    n = nsamp + wmax - 1
    view = _extended(fired, total, D + n).unfold(1, n, 1)
    chan = torch.arange(nchan, device="cuda")
    plane = torch.empty((ndm, n), dtype=torch.int32, device="cuda")
    start = torch.from_numpy(delay).cuda() + f0 % total
    for d in range(ndm):
        plane[d] = _root(view[chan, start[d]], mode, branching)
    return _candidates(plane, nsamp, widths, mode, f0), plane[:, wmax - 1:]


def _root(x, mode, branching):
    """The tree's root over [nchan][n] spikes: leaves of 4 channels, nodes of `branching` children."""
    if mode == "float":
        return x.sum(0, dtype=torch.int32)
    v, fan = x, 4
    while True:
        pad = -v.shape[0] % fan
        if pad:
            v = torch.cat([v, v.new_zeros((pad, v.shape[1]))])
        s = v.view(-1, fan, v.shape[1]).sum(1, dtype=torch.int32)
        v = (s >= 2).to(torch.uint8) if mode == "binary" else s.clamp_max(255).to(torch.uint8)
        if v.shape[0] == 1:
            return v[0].int()
        fan = branching


def _candidates(plane, nb, widths, mode, f0):
    ndm = plane.shape[0]
    y = plane.long()
    s1, s2 = y[:, :nb].sum(1).double(), (y[:, :nb] ** 2).sum(1).double()
    mu = s1 / nb
    sig = (s2 / nb - mu * mu).clamp_min(0).sqrt()
    if mode == "binary":
        sig = sig.clamp_min(0.2)
    csum = F.pad(y.cumsum(1), (1, 0))
    best = torch.full((ndm, nb), -1e300, dtype=torch.float64, device=y.device)
    width = torch.zeros((ndm, nb), dtype=torch.int32, device=y.device)
    for w in (1 << j for j in range(11)):
        rows = torch.tensor([d for d in range(ndm) if w in widths[d]], device=y.device, dtype=torch.long)
        if not len(rows):
            continue
        s = (csum[rows, w:w + nb] - csum[rows, :nb]).double()
        snr = (s - (mu[rows] * w)[:, None]) / (sig[rows] * math.sqrt(w))[:, None]
        up = snr > best[rows]
        best[rows] = torch.where(up, snr, best[rows])
        width[rows] = torch.where(up, torch.full_like(width[rows], w), width[rows])
        del s, snr, up
    mask = (best >= 7.0) & (sig > 0)[:, None]
    m = mask.float()[None, None]
    closed = 1 - F.max_pool2d(1 - F.max_pool2d(m, 9, 1, 4), 9, 1, 4)
    label = torch.arange(1, ndm * nb + 1, device=y.device, dtype=torch.float64).view(1, 1, ndm, nb) * closed
    while True:
        before = label
        for _ in range(32):
            label = F.max_pool2d(label, 3, 1, 1) * closed
        if torch.equal(label, before):
            break
    on = torch.nonzero(closed[0, 0].reshape(-1) > 0).reshape(-1)
    ids, npix = torch.unique(label.reshape(-1)[on], return_counts=True)
    npix = dict(zip(ids.tolist(), npix.tolist()))
    cell = torch.nonzero(mask.reshape(-1)).reshape(-1)
    lab, val, wid = (t.reshape(-1)[cell].cpu().numpy() for t in (label, best, width))
    cell = cell.cpu().numpy()
    out, seen = [], set()
    for i in np.lexsort((cell, -val.astype(np.float32))):
        if lab[i] in seen:
            continue
        seen.add(lab[i])
        if npix[lab[i]] >= 10:
            out.append((int(cell[i] % nb) + f0, int(cell[i] // nb), float(val[i]), int(wid[i]), npix[lab[i]]))
    return sorted(out)


def _exact_zfloat(case, chunks, fill):
    nchan, nsamp, ndm = case["nchan"], case["nsamp"], case["ndm"]
    delay = _delays(nchan, DT, np.linspace(0.0, case["dm_max"], ndm))
    D = int(delay.max())
    z = []
    for c in chunks:
        u, mu, sig = _levels(c, THETA["zfloat"])
        p = c.t().double()
        z.append(torch.where(p >= u[:, None], (p - mu[:, None]) / sig[:, None].clamp_min(1e-300), 0.0))
    z = torch.cat(z, 1)
    e0 = fill * nsamp - D
    view = _extended(z, z.shape[1], D + nsamp).unfold(1, nsamp, 1)
    start = torch.from_numpy(delay).cuda() + e0 % z.shape[1]
    chan = torch.arange(nchan, device="cuda")
    plane = torch.empty((ndm, nsamp), dtype=torch.float64, device="cuda")
    for d in range(ndm):
        plane[d] = view[chan, start[d]].sum(0)
    return plane / math.sqrt(nchan)


def _scrunch(case):
    """The rate factor of every trial DM: the largest power of two within the in-channel smearing."""
    f = _freqs(case["nchan"])
    df, fc = abs(f[1] - f[0]), (f[0] + f[-1]) / 2.0
    out = []
    for dm in np.linspace(0.0, case["dm_max"], case["ndm"]):
        s, tau = 1, K_DM * dm * df / fc ** 3
        while 2 * s <= case["s_max"] and 2 * s * DT <= tau:
            s *= 2
        out.append(s)
    return out


def _multirate_reach(case):
    return WMAX * max(_scrunch(case))


def _exact_multirate(case, chunks):
    fill = _history(case, _multirate_reach(case))[0]
    dms, scr = np.linspace(0.0, case["dm_max"], case["ndm"]), np.array(_scrunch(case))
    found = []
    for s in sorted(set(scr.tolist())):
        idx = np.nonzero(scr == s)[0]
        part = [((c.view(-1, s, c.shape[1]).int().sum(1) + s // 2) // s).to(torch.uint8) for c in chunks]
        for t, d, snr, w, npix in _search(case, part, fill, DT * s, dms[idx])[0]:
            found.append((t * s, int(idx[d]), snr, w * s, npix))
    parent = list(range(len(found)))

    def root(i):
        while parent[i] != i:
            i = parent[i]
        return i

    for i, a in enumerate(found):
        for j in range(i):
            b = found[j]
            if abs(dms[a[1]] - dms[b[1]]) <= 20.0 and abs(a[0] - b[0]) * DT <= 0.2:
                parent[root(i)] = root(j)
    best = {}
    for i, a in enumerate(found):
        r, key = root(i), (-np.float32(a[2]), a[1], a[0])
        if r not in best or key < best[r][0]:
            best[r] = (key, a)
    return sorted(v[1] for v in best.values())


def _exact_snippets(plane, rows, cols):
    r = rows[:, None, None] + torch.arange(-32, 32, device="cuda")[None, :, None]
    c = cols[:, None, None] + torch.arange(-128, 128, device="cuda")[None, None, :]
    out = torch.empty((len(rows), 64, 256), dtype=torch.float64, device="cuda")
    for i in range(0, len(rows), 256):
        ri, ci = r[i:i + 256], c[i:i + 256]
        ok = (ri >= 0) & (ri < plane.shape[0]) & (ci >= 0) & (ci < plane.shape[1])
        v = plane[ri.clamp(0, plane.shape[0] - 1), ci.clamp(0, plane.shape[1] - 1)].double()
        n = ok.sum((1, 2), keepdim=True)
        mu = (v * ok).sum((1, 2), keepdim=True) / n
        sig = (((v - mu) * ok) ** 2).sum((1, 2), keepdim=True).div(n).sqrt()
        out[i:i + 256] = torch.where(ok, (v - mu) / torch.where(sig > 0, sig, torch.ones_like(sig)), 0.0)
    return out


def _split_params(p):
    out, o = [], 0
    for shape in ((16, 1, 3, 3), (16,), (32, 16, 3, 3), (32,), (64, 32, 3, 3), (64,), (128, 16384), (128,), (1, 128),
                  (1,)):
        n = int(np.prod(shape))
        out.append(p[o:o + n].view(shape))
        o += n
    return out


def _network(x, w):
    h = x[:, None]
    for i in range(3):
        h = F.max_pool2d(F.relu(F.conv2d(h, w[2 * i], w[2 * i + 1], padding=1)), 2)
    h = F.relu(F.linear(h.flatten(1), w[6], w[7]))
    return F.linear(h, w[8], w[9])[:, 0]
